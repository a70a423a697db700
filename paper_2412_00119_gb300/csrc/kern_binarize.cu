// kern_binarize.cu -- MedianBinarization of real-valued input patterns
// (Alg. 1 l.5; Sec. 3.2: the median value is the threshold).
//
//   a_i = +1  iff  x_i > m,   m = the ceil(K/2)-th smallest of the pattern's K
//                              values (lower median), compared in fp32
//
// packed as bits (bit i % 64 of word i / 64 = 1 <-> +1, pad bits 0), the input
// format of bmlp_train / bmlp_predict.
//
// k_binarize_regs (K <= kRegMax): a warp, or two, per pattern, with the
// pattern's values in registers as order-preserving 32-bit keys (bits ^
// 0x80000000 for a clear sign bit, ~bits for a set one), so that memory is read
// once.  The median is the key p with #{key < p} <= rank < #{key <= p}.  It is
// bracketed: the median lies in [lo, hi], with #{key < lo} and #{key <= hi}
// known.  The smallest value is tried first (the median of image-like data, which
// is mostly zeros), then two of a sample of 32, then keys inside the bracket,
// interpolated linearly between its ends by the counts (from the sixth round on in turn with the middle of the
// key range, which alone ends after 32 rounds).  A round is one comparison per
// value and a warp sum.  Once at most 32 candidates are left a warp lists them,
// one per lane, and ranks each against the others; with many equal values the
// bracket's ends move onto values instead.  Then the values are compared with
// the median as floats, so -0 and +0 are equal as they are in fp32, and one
// ballot packs 32 of them.
// Bound: memory, then instructions (about 8 per value).  60,000 x 784 of
// grey levels: 36 us = 5.4 TB/s (the radix select 299 us), of normal values 82 (290).
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

constexpr int kRegMax = 64 * 64;

// kWarps warps per pattern (1, four patterns per CTA, or 2, a CTA), kR values per lane: K <= 32 kWarps kR;
// K >= 32 kWarps kFull, so the first kFull values of every lane are inside the
// pattern.  Value j of lane l of the pattern's warp w is x[32 (w + kWarps j) + l].
template <int kWarps, int kR, int kFull>
__global__ void __launch_bounds__(kWarps == 1 ? 128 : 32 * kWarps)
    k_binarize_regs(const float* __restrict__ x, int64_t n, int K, int nw, uint64_t* __restrict__ out) {
  constexpr int kPats = kWarps == 1 ? 4 : 1;     // patterns per CTA
  __shared__ uint32_t red[2][kWarps];
  __shared__ uint32_t cand[kPats][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = kWarps == 1 ? 0 : warp;
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
    for (int i = 1; i < kWarps; ++i)
      t = op == 0 ? t + red[flip][i] : (op == 1 ? min(t, red[flip][i]) : max(t, red[flip][i]));
    flip ^= 1;   // the next round writes the other buffer: no second barrier
    return t;
  };
  for (int64_t mu = (int64_t)blockIdx.x * kPats + (kWarps == 1 ? warp : 0); mu < n;
       mu += (int64_t)gridDim.x * kPats) {
    const float* row = x + mu * (int64_t)K;
    uint32_t key[kR];   // values past K: the largest key, never below a pivot
    auto inside = [&](int j) { return j < kFull || 32 * (w + kWarps * j) + lane < K; };
#pragma unroll
    for (int j = 0; j < kR; ++j)
      key[j] = inside(j) ? __float_as_uint(__ldcs(row + 32 * (w + kWarps * j) + lane)) : 0x7FFFFFFFu;
    uint32_t kmin = 0xFFFFFFFFu;
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      key[j] ^= (uint32_t)((int32_t)key[j] >> 31) | 0x80000000u;
      kmin = min(kmin, key[j]);
    }
    uint32_t lo = all_warps(kmin, 1), hi = 0xFFFFFFFFu;
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
      if (it == 0) {
        // not the smallest value: bracket between the 12th and the 21st of 32 values
        // from four places of the pattern, in key order (a bitonic sort over the lanes)
        uint32_t v = (lane & 2) ? ((lane & 1) ? key[7 * kR / 8] : key[5 * kR / 8])
                                : ((lane & 1) ? key[3 * kR / 8] : key[kR / 8]);
        if constexpr (kWarps > 1) {
          if (lane < 32 / kWarps) cand[0][32 / kWarps * warp + lane] = v;
          __syncthreads();
          v = cand[0][lane];
        }
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
          for (int j = k >> 1; j > 0; j >>= 1) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, v, j);
            v = ((lane & j) == 0) == ((lane & k) == 0) ? min(v, o) : max(v, o);
          }
        const uint32_t a = max(__shfl_sync(0xffffffffu, v, 11), lo), z = __shfl_sync(0xffffffffu, v, 20);
        uint32_t ca = 0u, cz = 0u;   // #{key < a}, #{key <= z}; z is a value or the padding
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          ca += key[j] < a ? 1u : 0u;
          cz += key[j] <= z ? 1u : 0u;
        }
        ca = all_warps(ca, 0);
        cz = z == 0xFFFFFFFFu ? (uint32_t)K : all_warps(cz, 0);
        if (rank < ca) {
          hi = a - 1u;
          chi = ca;
        } else {
          lo = a;
          clo = ca;
          if (rank < cz) {
            hi = z;
            chi = cz;
          } else {
            lo = z + 1u;
            clo = cz;
          }
        }
        if (lo >= hi) break;
      }
      if (chi - clo <= 32u && hi != 0xFFFFFFFFu) {
        // at most a warp of candidates: one per lane, ranked against the others
        uint32_t* list = cand[kWarps == 1 ? warp : 0];
        uint32_t at = 0u;   // where this warp's candidates go
        if constexpr (kWarps > 1) {
          uint32_t mine = 0u;
#pragma unroll
          for (int j = 0; j < kR; ++j) mine += (key[j] >= lo && key[j] <= hi) ? 1u : 0u;
          mine = __reduce_add_sync(0xffffffffu, mine);
          if (lane == 0) red[flip][warp] = mine;
          __syncthreads();
          for (int i = 0; i < warp; ++i) at += red[flip][i];
          flip ^= 1;
        }
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          const bool in = key[j] >= lo && key[j] <= hi;
          const unsigned b = __ballot_sync(0xffffffffu, in);
          if (in) list[at + __popc(b & ((1u << lane) - 1u))] = key[j];
          at += __popc(b);
        }
        if constexpr (kWarps > 1) __syncthreads();
        else __syncwarp();
        const uint32_t cnt = chi - clo;
        const uint32_t mine = (uint32_t)lane < cnt ? list[lane] : 0xFFFFFFFFu;
        uint32_t below = 0u;
        for (uint32_t i = 0; i < cnt; ++i) {
          const uint32_t o = list[i];
          below += (o < mine || (o == mine && i < (uint32_t)lane)) ? 1u : 0u;
        }
        const unsigned who = __ballot_sync(0xffffffffu, (uint32_t)lane < cnt && below == rank - clo);
        hi = __shfl_sync(0xffffffffu, mine, __ffs(who) - 1);
        if constexpr (kWarps > 1) __syncthreads();   // the list is the next pattern's
        else __syncwarp();
        break;
      }
      if (it >= 3 || chi - clo == 1u || hi == 0xFFFFFFFFu) {
        // the bracket's ends onto values (many equal ones, or one candidate)
        uint32_t a = 0xFFFFFFFFu, z = 0u;
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          if (key[j] >= lo) a = min(a, key[j]);
          if (key[j] <= hi && inside(j)) z = max(z, key[j]);
        }
        lo = all_warps(a, 1);
        hi = all_warps(z, 2);
        if (lo >= hi) break;
      }
      p = lo + ((hi - lo) >> 1);
      if (it < 6 || (it & 1) == 0) {
        const float flo = key_float(lo), fhi = key_float(hi);
        // eight values past the median, towards the farther end: the bracket then
        // closes from both sides, and soon holds at most a warp of candidates
        const float t = (float)(rank - clo) + 0.5f, na = (float)(chi - clo);
        const float to = 2.0f * t < na ? fminf(t + 8.0f, na - 0.5f) : fmaxf(t - 8.0f, 0.5f);
        const float f = flo + (fhi - flo) * (to / na);
        const uint32_t kf = float_key(f);
        if (kf >= lo && kf < hi) p = kf;   // (a NaN's or an infinity's key: the middle)
      }
    }
    // x > m as floats, on keys: none for a NaN m; m = -0 compares like +0; a NaN x
    // (keys above +infinity's; the padding is one) compares false
    const float m = key_float(hi);
    const uint32_t above = m == 0.0f ? 0x80000001u : (m == m ? hi + 1u : 0xFFFFFFFFu);
    const uint32_t width = above <= 0xFF800000u ? 0xFF800001u - above : 0u;
    // lane l holds words w + kWarps l and, beyond 32, w + kWarps (l + 32) of the row
    uint32_t mine[2] = {0u, 0u};
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      const unsigned bits = __ballot_sync(0xffffffffu, key[j] - above < width);
      if (lane == (j & 31)) mine[j >> 5] = bits;
    }
#pragma unroll
    for (int h = 0; h < (kR > 32 ? 2 : 1); ++h) {
      const int word = w + kWarps * (lane + 32 * h);
      if (word < 2 * nw) reinterpret_cast<uint32_t*>(out + mu * (int64_t)nw)[word] = mine[h];
    }
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
  // the fewest registers that hold the pattern; one warp as long as it can (a
  // round of two or more warps costs a barrier: 20,000 x 1200 normal values 107 us
  // with four warps a pattern)
  auto regs = [&](auto kern, int pats, int threads) {
    const int64_t ctas = (n + pats - 1) / pats;
    kern<<<(unsigned)(ctas < grid ? ctas : grid), threads, 0, st>>>(x, n, K, nw, out);
  };
  if (K <= 32 * 8) regs(k_binarize_regs<1, 8, 0>, 4, 128);
  else if (K <= 32 * 16) regs(k_binarize_regs<1, 16, 8>, 4, 128);
  else if (K <= 32 * 25) regs(k_binarize_regs<1, 25, 16>, 4, 128);
  else if (K <= 32 * 32) regs(k_binarize_regs<1, 32, 25>, 4, 128);
  else if (K <= 32 * 48) regs(k_binarize_regs<1, 48, 32>, 4, 128);
  else if (K <= 32 * 64) regs(k_binarize_regs<1, 64, 48>, 4, 128);
  else if (K <= 64 * 48) regs(k_binarize_regs<2, 48, 32>, 1, 64);
  else if (K <= kRegMax) regs(k_binarize_regs<2, 64, 48>, 1, 64);
  else k_binarize_median<<<(unsigned)grid, kBinThreads, 0, st>>>(x, n, K, nw, out);
}

}  // namespace bk
