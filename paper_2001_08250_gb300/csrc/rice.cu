// Compressed interest-vector deltas for GetUpdates (Section 7): the server
// sends its window of Bloom-filter deltas compressed.  The paper names no
// encoding; the library writes the Golomb-Rice code of the gaps between set
// bits: for set bits p_0 < p_1 < ..., gap_i = p_i - p_{i-1} - 1 (p_{-1} = -1)
// is written as (gap_i >> k) one-bits, a zero bit, then the k low bits of
// gap_i, least significant first; the stream is packed LSB-first (stream bit
// j = bit j % 8 of byte j / 8).  k defaults to floor(log2 g) for the mean gap
// g = (m - count) / count (0 when g = 0 or there are no set bits).
//
// Three kernels over blocks of 1024 words (one per thread): count the set bits
// (and zero the stream), which fixes k; per block, the first and last set bit
// and the code bits of its set bits after the first (those depend only on
// positions inside the block: a block max-scan of each word's last set bit
// gives the set bit before each word's first one), and the last block to finish
// scans the blocks for the set bit before each block and each block's first
// stream bit; per block, the codes are put together in shared memory and leave
// as whole words (only the block's first and last word are shared with its
// neighbours and OR-ed in).  A block whose codes do not fit shared memory (a
// given k far from the density) ORs them into the stream one by one.  A stream
// that would pass the buffer's end is reported (nbits = UINT64_MAX) and nothing
// is written past the end.
//
// Bound by the per-bit loops (integer instructions) and the launches.  16 Mi
// bits, a fifth of them set: 37 us a call among others, 59 for a first one alone
// (with two global atomics a code, a kernel for the scan and scratch from the
// default pool, which gives it back at every synchronisation: 69 and 261).
#include <cstdint>

#include "tpir_internal.h"

namespace tpir {
namespace {

constexpr int kRThreads = 1024;

struct RiceJob {
  const uint64_t* bits;
  uint64_t m;
  int32_t k;           // < 0: choose from the set-bit count
  uint32_t* out;       // cap_words 32-bit words
  uint64_t cap_words;
  uint64_t* result;    // nbits (or UINT64_MAX), count, k
};

__device__ __forceinline__ uint64_t r_word(const RiceJob& J, uint64_t w) {
  const uint64_t W = (J.m + 63) / 64;
  if (w >= W) return 0;
  uint64_t x = J.bits[w];
  const uint64_t rem = J.m - w * 64;
  if (rem < 64) x &= (1ull << rem) - 1;  // bits at or past m are ignored
  return x;
}

__device__ __forceinline__ void r_or(const RiceJob& J, uint64_t word, uint32_t v) {
  if (v && word < J.cap_words) atomicOr(J.out + word, v);
}

// stream bits [a, a + q) set to one
__device__ void r_ones(const RiceJob& J, uint64_t a, uint64_t q) {
  while (q) {
    const uint32_t off = static_cast<uint32_t>(a & 31);
    const uint32_t n = q < 32u - off ? static_cast<uint32_t>(q) : 32u - off;
    const uint32_t mask = (n == 32 ? 0xFFFFFFFFu : ((1u << n) - 1u)) << off;
    r_or(J, a >> 5, mask);
    a += n;
    q -= n;
  }
}

// the k low bits of v at stream bits [a, a + k)
__device__ void r_bits(const RiceJob& J, uint64_t a, uint64_t v, uint32_t k) {
  while (k) {
    const uint32_t off = static_cast<uint32_t>(a & 31);
    const uint32_t n = k < 32u - off ? k : 32u - off;
    const uint32_t piece = static_cast<uint32_t>(v & ((n == 32) ? 0xFFFFFFFFull : ((1ull << n) - 1)));
    r_or(J, a >> 5, piece << off);
    a += n;
    v >>= n;
    k -= n;
  }
}

template <typename T, typename Op>
__device__ __forceinline__ T r_block_scan(T x, T identity, Op op, T* warp_tot, T* block_total) {
  // inclusive scan within the warp, then across the warps' totals
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T v = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, v, d);
    if (lane >= d) v = op(v, y);
  }
  if (lane == 31) warp_tot[warp] = v;
  __syncthreads();
  if (warp == 0) {
    T t = lane < kRThreads / 32 ? warp_tot[lane] : identity;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const T y = __shfl_up_sync(0xFFFFFFFFu, t, d);
      if (lane >= d) t = op(t, y);
    }
    warp_tot[lane] = t;  // inclusive totals of warps 0..lane
  }
  __syncthreads();
  const T before = warp == 0 ? identity : warp_tot[warp - 1];
  const T incl = op(before, v);
  const T excl_in_warp = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
  const T excl = lane == 0 ? before : excl_in_warp;
  if (block_total) *block_total = warp_tot[kRThreads / 32 - 1];
  __syncthreads();
  return excl;
}

// Per-block values of the scan: first and last set bit of the block (-1 if
// none), code bits of the block's set bits after its first, then (from the
// scan) the set bit before the block, the block's first stream bit and its bits.
struct RiceBlock {
  long long first, last;
  unsigned long long inner;
  long long prev;
  unsigned long long off, len;
};

__device__ __forceinline__ uint32_t r_param(const RiceJob& J, uint64_t count) {
  if (J.k >= 0) return static_cast<uint32_t>(J.k);
  if (!count) return 0;
  const uint64_t g = (J.m - count) / count;
  return g ? 63u - static_cast<uint32_t>(__clzll(static_cast<long long>(g))) : 0u;
}

// 1: the stream zeroed, set bits counted (result[1] zeroed by the host)
__global__ void __launch_bounds__(kRThreads, 2) rice_count_kernel(const RiceJob J, uint32_t* ticket) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0u;
  const uint64_t W = (J.m + 63) / 64;
  const uint64_t w = blockIdx.x * (uint64_t)kRThreads + threadIdx.x;
  for (uint64_t i = w; i < J.cap_words; i += (uint64_t)gridDim.x * kRThreads) J.out[i] = 0u;
  unsigned long long c = w < W ? __popcll(r_word(J, w)) : 0ull;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) c += __shfl_down_sync(0xFFFFFFFFu, c, d);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(reinterpret_cast<unsigned long long*>(J.result + 1), c);
}

// Code bits of the set bits of x after its first one (gaps below 64).
__device__ __forceinline__ uint32_t r_tail_len(uint64_t x, uint32_t k) {
  uint32_t len = 0;
  if (x) {
    const uint32_t sh = k < 31 ? k : 31;
    uint64_t y = x & (x - 1);
    len = static_cast<uint32_t>(__popcll(static_cast<long long>(y))) * (1 + k);
    if (k < 6) {  // else the quotients of gaps below 64 are zero
      // (the two halves in turn: 32-bit operations)
      uint32_t p0 = static_cast<uint32_t>(__ffsll(static_cast<long long>(x)));
#pragma unroll
      for (uint32_t h = 0; h < 2; ++h) {
        uint32_t z = static_cast<uint32_t>(y >> (32 * h));
        while (z) {
          const uint32_t p = 32 * h + static_cast<uint32_t>(__ffs(static_cast<int>(z)));
          len += (p - p0 - 1) >> sh;
          p0 = p;
          z &= z - 1;
        }
      }
    }
  }
  return len;
}
__device__ __forceinline__ unsigned long long r_len(uint64_t gap, uint32_t k) { return (gap >> k) + 1 + k; }
__device__ __forceinline__ long long r_max(long long a, long long b) { return a > b ? a : b; }
__device__ __forceinline__ unsigned long long r_sum(unsigned long long a, unsigned long long b) { return a + b; }

// Scans the blocks (one CTA): the set bit before each block, its offset.
__device__ void r_scan_blocks(const RiceJob& J, RiceBlock* blocks, uint32_t nblocks, uint32_t k,
                              long long* s_max, unsigned long long* s_sum) {
  long long carry_prev = -1;
  unsigned long long carry_off = 0;
  for (uint32_t base = 0; base < nblocks; base += kRThreads) {
    const uint32_t b = base + threadIdx.x;
    RiceBlock blk{-1, -1, 0, -1, 0};
    if (b < nblocks) {  // written by other blocks of this launch: not through L1
      blk.first = __ldcg(&blocks[b].first);
      blk.last = __ldcg(&blocks[b].last);
      blk.inner = __ldcg(&blocks[b].inner);
    }
    long long chunk_last;
    long long prev = r_block_scan<long long>(blk.last, -1LL, r_max, s_max, &chunk_last);
    if (carry_prev > prev) prev = carry_prev;
    unsigned long long len = blk.inner;
    if (blk.first >= 0) len += r_len(static_cast<uint64_t>(blk.first - prev - 1), k);
    unsigned long long chunk_len;
    const unsigned long long off =
        carry_off + r_block_scan<unsigned long long>(len, 0ull, r_sum, s_sum, &chunk_len);
    if (b < nblocks) {
      blocks[b].prev = prev;
      blocks[b].off = off;
      blocks[b].len = len;
    }
    if (chunk_last > carry_prev) carry_prev = chunk_last;
    carry_off += chunk_len;
  }
  if (threadIdx.x == 0) {
    J.result[0] = carry_off <= J.cap_words * 32 ? carry_off : ~0ull;
    J.result[2] = k;
  }
}

// 2: per block (kRThreads words): first / last set bit, inner code bits; the
// last block to finish scans them
__global__ void __launch_bounds__(kRThreads, 2) rice_block_kernel(const RiceJob J, RiceBlock* blocks,
                                                               uint32_t* ticket) {
  __shared__ long long s_max[32];
  __shared__ unsigned long long s_sum[32];
  __shared__ long long s_first;
  __shared__ uint32_t s_last;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint64_t w = blockIdx.x * (uint64_t)kRThreads + threadIdx.x;
  const uint64_t x = r_word(J, w);  // (an input: not written by the kernel before)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const uint32_t k = r_param(J, J.result[1]);
  const long long last = x ? static_cast<long long>(w * 64 + 63 - __clzll(static_cast<long long>(x))) : -1;
  const long long first_here = x ? static_cast<long long>(w * 64 + __ffsll(static_cast<long long>(x)) - 1) : -1;
  if (threadIdx.x == 0) s_first = -1;
  long long block_last;
  const long long prev = r_block_scan<long long>(last, -1LL, r_max, s_max, &block_last);
  // the block's first set bit opens the first word with bits; its code needs
  // the set bit before the block and is left to the scan
  unsigned long long len = r_tail_len(x, k);
  if (x && prev >= 0) len += r_len(static_cast<uint64_t>(first_here - prev - 1), k);
  if (x && prev < 0) s_first = first_here;  // the word with bits whose prev is -1
  unsigned long long inner;
  r_block_scan<unsigned long long>(len, 0ull, r_sum, s_sum, &inner);
  if (threadIdx.x == 0) {
    blocks[blockIdx.x] = RiceBlock{s_first, block_last, inner, -1, 0, 0};
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  if (s_last) r_scan_blocks(J, blocks, gridDim.x, k, s_max, s_sum);
}

// 3: per block, the codes at the block's offset
constexpr uint32_t kRWindow = 6144;  // stream words put together in shared memory (24 KiB)
__global__ void __launch_bounds__(kRThreads, 2) rice_write_kernel(const RiceJob J, const RiceBlock* blocks) {
  __shared__ long long s_max[32];
  __shared__ unsigned long long s_sum[32];
  __shared__ uint32_t s_out[kRWindow];
  const uint64_t w = blockIdx.x * (uint64_t)kRThreads + threadIdx.x;
  const uint64_t x = r_word(J, w);  // (an input: not written by the kernels before)
  const long long last = x ? static_cast<long long>(w * 64 + 63 - __clzll(static_cast<long long>(x))) : -1;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const uint32_t k = r_param(J, J.result[1]);
  const RiceBlock blk = blocks[blockIdx.x];
  if (blk.len == 0) return;  // no set bits (uniform over the block)
  const uint64_t word0 = blk.off >> 5;
  const uint64_t words = ((blk.off + blk.len + 31) >> 5) - word0;  // stream words it touches
  const bool window = words <= kRWindow;
  if (window)
    for (uint32_t i = threadIdx.x; i < words; i += kRThreads) s_out[i] = 0u;
  long long prev = r_block_scan<long long>(last, -1LL, r_max, s_max, nullptr);
  if (blk.prev > prev) prev = blk.prev;
  unsigned long long len = 0;
  const uint64_t gap0 = x ? static_cast<uint64_t>(static_cast<long long>(w * 64 + __ffsll(static_cast<long long>(x)) - 1) - prev - 1) : 0;
  if (x) len = r_len(gap0, k) + r_tail_len(x, k);
  const unsigned long long off =
      blk.off + r_block_scan<unsigned long long>(len, 0ull, r_sum, s_sum, nullptr);
  if (window) {
    // (the scan's barriers stand between the zeroing and these)
    uint64_t a = off - (word0 << 5);  // bit within the window
    uint64_t acc = 0;                 // bits of the stream from word a0 on
    uint32_t a0 = static_cast<uint32_t>(a >> 5), fill = static_cast<uint32_t>(a & 31);
    uint64_t gap = gap0;
    uint32_t p0 = 0;
#pragma unroll 1
    for (uint32_t h = 0; h < 2; ++h) {
      uint32_t z = static_cast<uint32_t>(x >> (32 * h));
      while (z) {
        const uint32_t p = 32 * h + static_cast<uint32_t>(__ffs(static_cast<int>(z)));
        if (p0) gap = p - p0 - 1;  // (the word's first code has its own gap)
        p0 = p;
        z &= z - 1;
        uint64_t q = gap >> k;
        if (q < 16 && k < 16) {  // the usual code: at most 31 bits at once
          const uint32_t q32 = static_cast<uint32_t>(q);
          const uint32_t low = static_cast<uint32_t>(gap) & ((1u << k) - 1u);
          acc |= static_cast<uint64_t>(((1u << q32) - 1u) | (low << (q32 + 1))) << fill;
          fill += q32 + 1 + k;
          if (fill >= 32) {
            atomicOr(&s_out[a0++], static_cast<uint32_t>(acc));
            acc >>= 32;
            fill -= 32;
          }
          continue;
        }
        // q one bits and a zero, then the k low bits of the gap, through a 64-bit
        // register whose full words are OR-ed out
        while (q >= 32) {
          acc |= 0xFFFFFFFFull << fill;
          atomicOr(&s_out[a0++], static_cast<uint32_t>(acc));
          acc >>= 32;
          q -= 32;
        }
        acc |= ((1ull << q) - 1) << fill;
        fill += static_cast<uint32_t>(q) + 1;
        if (fill >= 32) {
          atomicOr(&s_out[a0++], static_cast<uint32_t>(acc));
          acc >>= 32;
          fill -= 32;
        }
        uint64_t low = k ? gap & ((1ull << k) - 1) : 0;
        uint32_t kk = k;
        while (kk) {
          const uint32_t n = kk < 32 ? kk : 32;
          acc |= (low & ((1ull << n) - 1)) << fill;
          fill += n;
          if (fill >= 32) {
            atomicOr(&s_out[a0++], static_cast<uint32_t>(acc));
            acc >>= 32;
            fill -= 32;
          }
          low >>= n;
          kk -= n;
        }
      }
    }
    if (fill && acc) atomicOr(&s_out[a0], static_cast<uint32_t>(acc));
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < words; i += kRThreads) {
      if (i == 0 || i == words - 1)
        r_or(J, word0 + i, s_out[i]);
      else if (word0 + i < J.cap_words)
        J.out[word0 + i] = s_out[i];
    }
    return;
  }
  long long p0 = prev;
  uint64_t y = x, a = off;
  while (y) {
    const long long p = static_cast<long long>(w * 64 + __ffsll(static_cast<long long>(y)) - 1);
    const uint64_t gap = static_cast<uint64_t>(p - p0 - 1);
    const uint64_t q = gap >> k;
    r_ones(J, a, q);
    a += q + 1;  // the zero bit stays zero
    if (k) r_bits(J, a, gap, k);
    a += k;
    p0 = p;
    y &= y - 1;
  }
}

}  // namespace

size_t rice_scratch_bytes(uint64_t m) {
  const uint64_t W = (m + 63) / 64;
  return ((W + kRThreads - 1) / kRThreads) * sizeof(RiceBlock) + 16;  // the blocks, then the ticket
}

cudaError_t launch_rice_encode(const RiceRequest& q, void* scratch, cudaStream_t st) {
  const uint64_t W = (q.m + 63) / 64;
  const uint64_t nb = (W + kRThreads - 1) / kRThreads;
  if (nb == 0 || nb > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  const RiceJob J{q.bits, q.m, q.k, q.out, q.cap_words, q.result};
  RiceBlock* blocks = static_cast<RiceBlock*>(scratch);
  uint32_t* ticket = reinterpret_cast<uint32_t*>(blocks + nb);
  cudaError_t e = cudaMemsetAsync(q.result, 0, 3 * sizeof(uint64_t), st);
  if (e != cudaSuccess) return e;
  const dim3 grid(static_cast<uint32_t>(nb)), block(kRThreads);
  rice_count_kernel<<<grid, block, 0, st>>>(J, ticket);
  count_launches();
  e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_pdl(rice_block_kernel, grid, block, 0, st, J, blocks, ticket);
  if (e == cudaSuccess)
    e = launch_pdl(rice_write_kernel, grid, block, 0, st, J, static_cast<const RiceBlock*>(blocks));
  return e;
}

}  // namespace tpir
