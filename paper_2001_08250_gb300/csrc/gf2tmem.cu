// Tensor-core form of the batched PIR read (Section 2 step 5, batched as in
// Section 9.2): Out = R (x) T over GF(2).  Each output bit is the parity of
// an integer: the number of buckets k with request bit R[b][k] = 1 and table
// bit T[k][c] = 1.  The kernel computes these integers exactly as a product
// of 0/1 matrices on the 5th-generation tensor cores and keeps the low bit of
// each: exactly the XOR of the selected buckets, with every bucket read for
// every request as in the scalar kernels.
//
// Operands.  Both matrices are packed 4-bit e2m1 values in the block-scaled
// MMA (tcgen05.mma kind::mxf4, every scale factor 1.0 = UE8M0 0x7F),
// accumulated in fp32 in tensor memory: every product is 0 or 1.0 and a
// k-chunk's counts stay far below 2^23, exact in fp32.  A table nibble
// is the bit where it stands (0.5, 1.0 or 2.0 by its place in the nibble; the
// fourth place is shifted to 2.0) and the request nibble of the same bucket
// holds the inverse, so that a table word of 32 bits becomes its 32 nibbles
// with four ANDs and one shift.
//
// Roles of the operands.  The table is the M side (128 table columns of the
// bit-transposed copy, tcopy.cu) and lives in tensor memory: each expander
// thread owns one column (one tensor-memory lane) and writes its nibbles with
// tcgen05.st, so the operand that changes with every MMA costs no
// shared-memory stores and no shared-memory operand reads.  The requests are the N
// side (up to 128 a block): the nibbles of one k-chunk of the block are
// expanded into shared memory once per item and stay there while the item's
// column tiles stream past.  Per MMA (M = 128 columns x N requests x K = 64
// buckets) shared memory carries only the N operand's read (32 N bytes) and
// the 1 KiB of raw table words in and out.
//
// An item is (block of up to 128 requests, k-chunk of kc_words x 64 buckets, run
// of column tiles).  A CTA (persistent, one per SM) runs two streams of tiles
// side by side, each with its own raw ring, tensor-memory ring, MMA issuer and
// accumulator(s): asking a barrier takes about 90 clocks, issuing an MMA 25 to
// 50 and a committed stage some 300 to be handed back, and with one stream
// these hand-offs bounded the read (82 us at 128 requests of 32 768 x 4 KiB,
// against 45 with two; the MMAs alone take 28).
//   warps 0, 1    stream the raw stages: 4 words (256 buckets) of a tile's 128
//                 columns by 2-D TMA;
//   warps 2, 3    issue the MMAs;
//   8 or 16 warps table expanders, one or two groups of four per stream (lane
//                 quarter = warp % 4; TLayout);
//   8 warps       expand the item's requests, then take the tiles in order:
//                 read the counts (tcgen05.ld), keep their parities, transpose
//                 them into reply words, and store or XOR-reduce those.
// Tensor memory: per stream one accumulator of 128 (or 112) columns (used as
// two where no block holds more than 64 (or 48) requests) and three (or four)
// table stages of 32 columns; the scale factors in the last 32.  Every wait is
// bounded; a wait that gives up sets the status word, and the CTA drains its MMAs
// and TMA loads and frees its tensor memory before it returns.
//
// Measured (us a launch; before: both operands in shared memory, one CTA an
// SM): 32 768 x 4 KiB: 33 at 32 requests (68 on the register-tiled kernel), 36
// at 64 (77), 42 at 112, 44 at 128 (77); 50 021 x 4 160 bytes masked: 65 at 100
// requests (134); 200 003 x 128 bytes: 12.5 at 64 (93 on the register-tiled
// kernel).  Blocks of up to 112 requests with one expander group: 39, 40, 44 and
// 80, 12.4.  What bounds it: instruction latency and the ALU pipe in the
// expanders and the issuers (issue slots 57 % used, ALU pipe 54 %, tensor pipe 56 %
// at 128 requests; HBM 60 % at 32).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "bits.cuh"
#include "chacha.cuh"
#include "mbar.cuh"
#include "tpir_internal.h"

namespace tpir {
namespace {

constexpr uint32_t kTCols = 128;               // table columns per tile (MMA M)
constexpr uint32_t kTStageWords = 4;           // 64-bucket words per stage
constexpr uint32_t kTRawBytes = kTCols * kTStageWords * 8;  // 4 KiB
constexpr uint32_t kTStreams = 2;              // independent tile pipelines of a CTA
constexpr uint32_t kTMaxN = 128;               // requests per block
constexpr uint32_t kTAccHalf = 64;             // columns to a stream's second accumulator
constexpr uint32_t kTSlotCols = 8 * kTStageWords;
constexpr uint32_t kTOutBytes = 128 * 16;      // a tile's reply words: 16 bytes per request
constexpr uint32_t kTSfa = 480, kTSfb = 496;   // scale factors
constexpr uint32_t kTTmemCols = 512;
constexpr uint32_t kTIssueWarp0 = kTStreams;   // after one TMA warp per stream
constexpr uint32_t kTExpWarp0 = 2 * kTStreams;
constexpr uint32_t kTEpiWarps = 8;
static_assert(kTExpWarp0 % 4 == 0, "a warp reads the tensor-memory lanes of its quarter");

// The two layouts of a CTA (with one group a stage's expansion, some 600 clocks
// of dependent instructions, bounded the blocks that the MMAs do not).  G = 1: blocks of up to 128 requests, one group of
// four expander warps per stream.  G = 2: blocks of up to 112 requests, whose
// accumulators leave room for a fourth table stage per stream, and two groups
// that take alternate stages; the rings are of even length, so that a slot
// always belongs to the same group.
template <int G>
struct TLayout {
  static constexpr uint32_t kRaw = G == 1 ? 5 : 6;           // raw stages in flight, per stream
  static constexpr uint32_t kSlots = G == 1 ? 3 : 4;         // table stages in tensor memory, per stream
  static constexpr uint32_t kAcc = G == 1 ? 128 : 112;       // accumulator columns per stream
  static constexpr uint32_t kRes = (G == 1 ? 176 : 168) * 1024;  // expanded requests of an item
  static constexpr uint32_t kACol = kTStreams * kAcc;        // first column of the table rings
  static constexpr uint32_t kEpiWarp0 = kTExpWarp0 + 4 * G * kTStreams;
  static constexpr int kThreads = 32 * (kEpiWarp0 + kTEpiWarps);
  static constexpr uint32_t kOut0 = kRes + kTStreams * kRaw * kTRawBytes;
  static constexpr uint32_t kSmem = 1024 + kOut0 + 2 * kTOutBytes;
  static_assert(kSmem <= 231424, "dynamic shared memory above 227 KiB less the static part");
  static_assert(kACol + kTStreams * kSlots * kTSlotCols <= kTSfa, "tensor memory columns overlap");
  static_assert(kRaw % G == 0 && kSlots % G == 0, "a ring slot belongs to one group");
};
constexpr uint64_t kTWaitNs = 4000000000ull;

struct TJob {
  const uint64_t* R;
  uint32_t* out;
  const uint8_t* seeds;  // masks of a serialized-PIR read, or null
  uint64_t n;
  uint32_t Wd, words64, B;
  uint32_t nw;           // request words of the job's own buckets: ceil(n / 64)
  uint32_t tiles;        // column tiles: Wd / 4
  uint32_t mbs, mb_rows; // request blocks, requests per block (a multiple of 16)
  uint32_t kcs, kc_words;
  uint32_t splits;       // column tiles t, t + splits, ... form one item
  uint32_t item_begin;
  uint32_t split;        // 0: replies stored; 1: initialised first (zeros or masks), XOR-reduced
                         // into; 2: masked, stored by their single writer with the mask
};

template <int NJ>
struct TLaunch {
  CUtensorMap maps[NJ];
  TJob jobs[NJ];
  uint32_t njobs, total_items;
  uint32_t nbuf;  // accumulators per stream: 2 when every job's blocks fit half of one
};
constexpr int kTMultiJobs = 64;  // jobs per many-table launch (kernel parameter space)
static_assert(sizeof(TLaunch<kTMultiJobs>) <= 32000, "kernel parameters must stay below 32 KB");

struct TItem {
  uint32_t job, b0, w0, w1;  // requests from b0, words [w0, w1)
  uint32_t t0, nt;           // tiles t0, t0 + splits, ... (nt of them)
};

// The r-th item of this CTA (items are listed by descending cost; alternate
// rounds sweep the grid in alternate directions).  Request blocks fastest, so
// that the CTAs of a round share the table words in L2.
template <int NJ>
__device__ __forceinline__ bool t_item(const TLaunch<NJ>& L, uint32_t r, TItem& it) {
  const uint32_t c = (r & 1u) ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
  const uint32_t item = c + r * gridDim.x;
  if (item >= L.total_items) return false;
  uint32_t lo = 0;
  if constexpr (NJ > 1) {
    uint32_t hi = L.njobs - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (L.jobs[mid].item_begin <= item)
        lo = mid;
      else
        hi = mid - 1;
    }
  }
  const TJob& J = L.jobs[lo];
  uint32_t local = item - J.item_begin;
  it.job = lo;
  it.b0 = (local % J.mbs) * J.mb_rows;
  local /= J.mbs;
  it.t0 = local % J.splits;
  it.nt = (J.tiles - it.t0 + J.splits - 1) / J.splits;
  it.w0 = (local / J.splits) * J.kc_words;
  it.w1 = min(J.nw, it.w0 + J.kc_words);
  return true;
}

// Shared-memory matrix descriptor of one K = 64 step of the N operand: K-major
// without swizzle, 8-row x 16-byte core matrices, 128 bytes apart along K, 256
// along N; the steps of a chunk are 32 N bytes apart.
// (The lower half holds the address and the distance along K.)
constexpr uint32_t kTDescHi = (256u >> 4) | (1u << 14);
__device__ __forceinline__ uint32_t t_desc(uint32_t addr) {
  return ((addr >> 4) & 0x3FFFu) | (static_cast<uint32_t>(128 >> 4) << 16);
}

// D (+)= A x B.  Whether D is accumulated is a compile-time constant: back to
// back and with fixed operands an MMA then takes its thread 12 clocks to issue,
// 51 with the predicate formed at run time.
template <bool ACC>
__device__ __forceinline__ void t_mma(uint32_t d, uint32_t a, uint32_t bdesc, uint32_t idesc,
                                      uint32_t sfa, uint32_t sfb) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 q;\n\tsetp.ne.b32 p, %7, 0;\n\tmov.b64 q, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], q, %4, [%5], [%6], "
      "p;\n\t}" ::"r"(d),
      "r"(a), "r"(bdesc), "r"(kTDescHi), "r"(idesc), "r"(sfa), "r"(sfb), "n"(ACC ? 1 : 0)
      : "memory");
}

__device__ __forceinline__ void t_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   mb::saddr(bar))
               : "memory");
}

// One thread of the (converged) warp.
__device__ __forceinline__ bool t_elect() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(p));
  return p != 0;
}
// mb::wait by a whole warp, every branch taken by all of it (the votes), so
// that the compiler keeps the caller's loop state in uniform registers.
__device__ __forceinline__ bool t_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                            int* status) {
  if (__all_sync(0xFFFFFFFFu, mb::try_wait(bar, parity))) return true;
  const uint64_t t0 = mb::gtimer();
  while (!__all_sync(0xFFFFFFFFu, mb::try_wait(bar, parity))) {
    const bool late = mb::gtimer() - t0 > kTWaitNs;
    if (__any_sync(0xFFFFFFFFu, late)) {
      *abort_flag = 1;
      atomicExch(status, static_cast<int>(TPIR_ETIMEDOUT));
      return false;
    }
    if (__any_sync(0xFFFFFFFFu, *abort_flag != 0)) return false;
  }
  return true;
}

// 32 buckets' request bits as 32 nibbles: nibble m of word t is bucket 4 m + t
// of the chunk, with the inverse of the table nibble's value (t_table_words).
__device__ __forceinline__ uint4 t_request_words(uint32_t h) {
  return make_uint4((h << 2) & 0x44444444u, h & 0x22222222u, (h >> 2) & 0x11111111u,
                    (h >> 3) & 0x11111111u);
}

// This thread's tensor-memory lane: 32 columns (256 nibbles) at taddr from
// the four 64-bucket words of its table column.
__device__ __forceinline__ void t_store_stage(uint32_t taddr, const uint64_t (&x)[4]) {
  uint32_t v[32];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t w = static_cast<uint32_t>(x[i] >> (32 * h));
      v[8 * i + 4 * h] = w & 0x11111111u;           // 0.5
      v[8 * i + 4 * h + 1] = w & 0x22222222u;       // 1.0
      v[8 * i + 4 * h + 2] = w & 0x44444444u;       // 2.0
      v[8 * i + 4 * h + 3] = (w >> 1) & 0x44444444u;  // 2.0
    }
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
      "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]),
      "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]),
      "r"(v[30]), "r"(v[31])
      : "memory");
}

// The four words of this thread's column in a raw stage.
__device__ __forceinline__ void t_read_raw(uint32_t addr, uint64_t (&x)[4]) {
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i)
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(x[i]) : "r"(addr + i * (kTCols * 8)) : "memory");
}

// 32 accumulator columns of this thread's lane (in registers after t_wait_ld).
__device__ __forceinline__ void t_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void t_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// Their parities: bit j = column j.  A count plus 2^23 has the count in its
// mantissa; the funnel shift takes its lowest bit.
__device__ __forceinline__ uint32_t t_parities(const uint32_t (&r)[32]) {
  uint32_t w = 0;
#pragma unroll
  for (int j = 0; j < 32; ++j)
    w = __funnelshift_r(w, __float_as_uint(__uint_as_float(r[j]) + 8388608.0f), 1);
  return w;
}

// The item's requests into shared memory: rows b0 .. b0 + mb_rows - 1 (zeros
// past the batch), words w0 .. w1 - 1, by the reply warps (this one: w).  A warp
// takes 8 requests x 4 words at a time, lane = 8 word + request: each load
// touches eight 32-byte sectors (a lane per request and four words a lane
// touched 32, and the load of a full block took 9 000 clocks), each quarter
// warp's store is 128 contiguous bytes; the loads of six such groups are in
// flight together.
__device__ __forceinline__ void t_load_requests(const TJob& J, const TItem& it, uint32_t res0,
                                                uint32_t w, uint32_t lane) {
  constexpr uint32_t kBatch = 6;
  const uint32_t N = J.mb_rows, W = it.w1 - it.w0, n8 = N / 8;
  const uint32_t groups = n8 * ((W + 3) / 4);
  const uint32_t r8 = lane & 7u, j = lane >> 3;
  for (uint32_t i0 = w; i0 < groups; i0 += kBatch * kTEpiWarps) {
    uint64_t x[kBatch];
#pragma unroll
    for (uint32_t c = 0; c < kBatch; ++c) {
      const uint32_t i = i0 + c * kTEpiWarps, b = it.b0 + (i % n8) * 8 + r8, k = (i / n8) * 4 + j;
      x[c] = 0;
      if (i < groups && b < J.B && k < W) x[c] = __ldg(J.R + static_cast<uint64_t>(b) * J.words64 + it.w0 + k);
    }
#pragma unroll
    for (uint32_t c = 0; c < kBatch; ++c) {
      const uint32_t i = i0 + c * kTEpiWarps, k = (i / n8) * 4 + j;
      if (i < groups && k < W) {
        const uint32_t o = res0 + k * (32 * N) + (i % n8) * 256u + r8 * 16u;
        const uint4 lo = t_request_words(static_cast<uint32_t>(x[c]));
        const uint4 hi = t_request_words(static_cast<uint32_t>(x[c] >> 32));
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(o), "r"(lo.x), "r"(lo.y),
                     "r"(lo.z), "r"(lo.w)
                     : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(o + 128u), "r"(hi.x), "r"(hi.y),
                     "r"(hi.z), "r"(hi.w)
                     : "memory");
      }
    }
  }
}

// Words w and w + 1 (w even) of the mask with this seed: words w % 16 and the next
// of ChaCha20 block w / 16, by selects (an index not known at compile time would
// send the block to local memory).
__device__ __noinline__ uint64_t t_mask(const uint8_t* seed, uint32_t w) {
  const uint4 ka = __ldg(reinterpret_cast<const uint4*>(seed)), kb = __ldg(reinterpret_cast<const uint4*>(seed) + 1);
  const uint32_t key[8] = {ka.x, ka.y, ka.z, ka.w, kb.x, kb.y, kb.z, kb.w};
  uint32_t k[16];
  cc_block(key, w >> 4, k);
  uint32_t lo = k[0], hi = k[1];
#pragma unroll
  for (uint32_t i = 2; i < 16; i += 2) {
    lo = (w & 15u) == i ? k[i] : lo;
    hi = (w & 15u) == i ? k[i + 1] : hi;
  }
  return lo | static_cast<uint64_t>(hi) << 32;
}

template <int NJ, int G>
__global__ void __launch_bounds__(TLayout<G>::kThreads, 1)
    gf2_tmem_kernel(const __grid_constant__ TLaunch<NJ> L, int* status) {
  using Y = TLayout<G>;
  constexpr uint32_t kTRaw = Y::kRaw, kTSlots = Y::kSlots, kTACol = Y::kACol, kTEpiWarp0 = Y::kEpiWarp0;
  constexpr uint32_t kTResBytes = Y::kRes, kTOut0 = Y::kOut0, kTAcc = Y::kAcc;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kTStreams][kTSlots], empty[kTStreams][kTSlots];
  __shared__ __align__(8) uint64_t raw_full[kTStreams][kTRaw], raw_empty[kTStreams][kTRaw];
  __shared__ __align__(8) uint64_t accf[kTStreams][2], acce[kTStreams][2], drain[kTStreams];
  __shared__ __align__(8) uint64_t reqf, reqe, outf;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t res0 = mb::saddr(base);
  volatile int* abort_flag = &s_abort;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (uint32_t g = 0; g < kTStreams; ++g) {
      for (uint32_t s = 0; s < kTSlots; ++s) {
        mb::init(&full[g][s], 4);  // the stream's four expander warps
        mb::init(&empty[g][s], 1);
      }
      for (int b = 0; b < 2; ++b) {
        mb::init(&accf[g][b], 1);
        mb::init(&acce[g][b], kTEpiWarps);
      }
      mb::init(&drain[g], 1);
      for (uint32_t s = 0; s < kTRaw; ++s) {
        mb::init(&raw_full[g][s], 1);
        mb::init(&raw_empty[g][s], 4);
      }
    }
    mb::init(&reqf, kTEpiWarps);
    mb::init(&reqe, kTStreams);
    mb::init(&outf, kTEpiWarps);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kTEpiWarp0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     mb::saddr(&s_tmem)),
                 "r"(kTTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  if (warp >= kTEpiWarp0 && warp < kTEpiWarp0 + 4) {
    // scale factors of every MMA: UE8M0 1.0 in columns 480..511 of all lanes
    const uint32_t one = 0x7F7F7F7Fu;
    for (uint32_t col = kTSfa; col < kTTmemCols; col += 8)
      asm volatile(
          "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(
              tmem + (((warp & 3u) * 32u) << 16) + col),
          "r"(one)
          : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (warp < kTStreams) {
    // ---------------- raw table words of stream `warp` (TMA) ----------------
    const uint32_t g = warp, raw0 = res0 + kTResBytes + g * (kTRaw * kTRawBytes);
    if (lane == 0) {
      uint32_t p = 0;
      TItem it;
      bool ok = true;
      for (uint32_t r = 0; ok && t_item(L, r, it); ++r) {
        const uint64_t map = reinterpret_cast<uint64_t>(&L.maps[it.job]);
        const uint32_t tstep = L.jobs[it.job].splits;
        for (uint32_t i = g; ok && i < it.nt; i += kTStreams) {
          const uint32_t t = it.t0 + i * tstep;
          for (uint32_t w = it.w0; w < it.w1; w += kTStageWords, ++p) {
            const uint32_t rs = p % kTRaw, ph = (p / kTRaw) & 1u;
            if (!mb::wait_sleep(&raw_empty[g][rs], ph ^ 1u, abort_flag, status, kTWaitNs, 32)) {
              ok = false;
              break;
            }
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                             mb::saddr(&raw_full[g][rs])),
                         "r"(kTRawBytes)
                         : "memory");
            // 4 words of the tile's 128 columns (zeros past the table)
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                "[%0], [%1, {%2, %3}], [%4];" ::"r"(raw0 + rs * kTRawBytes),
                "l"(map), "r"(static_cast<int>(t * kTCols)), "r"(static_cast<int>(w)),
                "r"(mb::saddr(&raw_full[g][rs]))
                : "memory");
          }
        }
      }
      // Loads still landing (an aborted run) complete before the CTA exits: a
      // slot has at most one load in flight, its latest.
      for (uint32_t rs = 0; rs < kTRaw && rs < p; ++rs) {
        const uint32_t last = rs + kTRaw * ((p - 1 - rs) / kTRaw);
        const uint64_t t0 = mb::gtimer();
        while (!mb::try_wait(&raw_full[g][rs], (last / kTRaw) & 1u)) {
          if (mb::gtimer() - t0 > kTWaitNs) {
            atomicExch(status, static_cast<int>(TPIR_ETIMEDOUT));
            break;
          }
        }
      }
    }
  } else if (warp < kTExpWarp0) {
    // ------------------------- MMA issue of one stream -------------------------
    // The whole warp walks the stages, one elected thread issues: an MMA costs
    // its thread fewer clocks than in a loop inside `if (lane == 0)` (55 against
    // 93).
    const uint32_t g = __shfl_sync(0xFFFFFFFFu, warp, 0) - kTIssueWarp0;
    const bool one = t_elect();
    const uint32_t utmem = __shfl_sync(0xFFFFFFFFu, tmem, 0);
    const uint32_t sfa = utmem + kTSfa, sfb = utmem + kTSfb;
    const uint32_t a0 = utmem + kTACol + g * (kTSlots * kTSlotCols);
    const uint32_t bd0 = t_desc(__shfl_sync(0xFFFFFFFFu, res0, 0));
    const uint32_t nb2 = L.nbuf == 2 ? 1u : 0u;
    uint32_t is = 0, iph = 0;  // ring slot and its phase
    uint32_t tc = 0;           // this stream's tiles so far
    TItem it;
    bool ok = true;
    for (uint32_t r = 0; ok && t_item(L, r, it); ++r) {
      const uint32_t N = L.jobs[it.job].mb_rows;
      // A and B e2m1 (1), both K-major, UE8M0 scales (bit 23), M = 128
      const uint32_t idesc = (1u << 7) | (1u << 10) | ((N >> 3) << 17) | (1u << 23) | ((128u >> 4) << 24);
      const uint32_t dstep = (32u * N) >> 4;
      if (!t_wait_warp(&reqf, r & 1u, abort_flag, status)) break;
      // (an issuer without a tile in this item says so too: the next phase of
      // reqf completes only after both have seen this one)
      if (one) mb::arrive(&reqe);
      const uint32_t W = it.w1 - it.w0;
      for (uint32_t i = g; ok && i < it.nt; i += kTStreams, ++tc) {
        const uint32_t buf = nb2 & tc, acc = utmem + g * kTAcc + buf * kTAccHalf;
        const uint32_t use = tc >> nb2;  // times this accumulator was used before
        if (use && !t_wait_warp(&acce[g][buf], (use - 1u) & 1u, abort_flag, status)) {
          ok = false;
          break;
        }
        uint32_t bd = bd0;
        for (uint32_t w = 0; w < W; w += kTStageWords) {
          if (!t_wait_warp(&full[g][is], iph, abort_flag, status)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t s = is, a = a0 + s * kTSlotCols, nk = min(kTStageWords, W - w);
          if (++is == kTSlots) {
            is = 0;
            iph ^= 1u;
          }
          if (one) {
            if (w)
              t_mma<true>(acc, a, bd, idesc, sfa, sfb);
            else
              t_mma<false>(acc, a, bd, idesc, sfa, sfb);
#pragma unroll
            for (uint32_t j = 1; j < kTStageWords; ++j)
              if (j < nk) t_mma<true>(acc, a + 8 * j, bd + j * dstep, idesc, sfa, sfb);
            t_commit(&empty[g][s]);
          }
          __syncwarp();
          bd += kTStageWords * dstep;
        }
        if (ok && one) t_commit(&accf[g][buf]);
        __syncwarp();
      }
    }
    // Drain: every MMA issued completes before the tensor memory is freed.
    if (one) {
      t_commit(&drain[g]);
      const uint64_t t0 = mb::gtimer();
      while (!mb::try_wait(&drain[g], 0)) {
        if (mb::gtimer() - t0 > kTWaitNs) {
          atomicExch(status, static_cast<int>(TPIR_ETIMEDOUT));
          break;
        }
      }
    }
    __syncwarp();
  } else if (warp < kTEpiWarp0) {
    // ------------------------ table expanders ------------------------
    // lane = column 32 quarter + lane of the tile; every stage is expanded in
    // full (words past the chunk are not multiplied)
    const uint32_t e = (warp - kTExpWarp0) >> 2, g = e % kTStreams, group = e / kTStreams, quarter = warp & 3u;
    const uint32_t raw0 = res0 + kTResBytes + g * (kTRaw * kTRawBytes) + (32u * quarter + lane) * 8u;
    const uint32_t tlane = tmem + ((32u * quarter) << 16) + kTACol + g * (kTSlots * kTSlotCols);
    uint32_t total = 0;  // the stream's stages
    TItem it;
    for (uint32_t r = 0; t_item(L, r, it); ++r)
      total += ((it.nt + kTStreams - 1 - g) / kTStreams) *
               ((it.w1 - it.w0 + kTStageWords - 1) / kTStageWords);
    // One set of warps waits for every phase of a ring slot in order (a phase's
    // parity says nothing while the phase before it is still open).  The next
    // stage's barriers are asked and its words read while this one is stored:
    // asking takes about 90 clocks, and in turn they bounded the pipeline.
    uint32_t rs = group, rph = 0, sl = group, ph = 0;  // ring slots and their phases
    bool slot_ready = false, ok = true;
    uint64_t x[4];
    if (group < total) {
      ok = mb::wait(&raw_full[g][rs], 0, abort_flag, status, kTWaitNs);
      t_read_raw(raw0 + rs * kTRawBytes, x);
    }
    for (uint32_t m = group; ok && m < total; m += G) {
      __syncwarp();
      // the raw slot goes back once the words are in registers and ordered
      // before the async proxy's next write to it
      asm volatile("fence.proxy.async.shared::cta;" ::"l"(x[0]), "l"(x[1]), "l"(x[2]), "l"(x[3]) : "memory");
      __syncwarp();
      if (lane == 0) mb::arrive(&raw_empty[g][rs]);
      if ((rs += G) >= kTRaw) {
        rs -= kTRaw;
        rph ^= 1u;
      }
      const bool more = m + G < total;
      const bool next = more && mb::test(&raw_full[g][rs], rph);
      if (!slot_ready && !mb::wait(&empty[g][sl], ph ^ 1u, abort_flag, status, kTWaitNs)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      __syncwarp();
      t_store_stage(tlane + sl * kTSlotCols, x);
      if (next) t_read_raw(raw0 + rs * kTRawBytes, x);
      const uint32_t s0 = sl;
      if ((sl += G) >= kTSlots) {
        sl -= kTSlots;
        ph ^= 1u;
      }
      slot_ready = mb::test(&empty[g][sl], ph ^ 1u);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mb::arrive(&full[g][s0]);
      if (more && !next) {
        if (!mb::wait(&raw_full[g][rs], rph, abort_flag, status, kTWaitNs)) break;
        t_read_raw(raw0 + rs * kTRawBytes, x);
      }
    }
  } else {
    // ---------------- requests in, replies out ----------------
    // The eight warps take the tiles in order, the streams in turn: warp
    // (quarter, half) reads its 32 table columns' counts for half of the
    // requests (two warps a column keep an accumulator occupied for half the
    // time), and the reply words of the four quarters meet in shared memory, so
    // that each request's 16 bytes leave in one sector.
    const uint32_t quarter = warp & 3u, half = ((warp - kTEpiWarp0) >> 2) & 1u;
    const uint32_t et = threadIdx.x - 32 * kTEpiWarp0;
    const uint32_t out0 = res0 + kTOut0;
    const uint32_t nb2 = L.nbuf == 2 ? 1u : 0u;
    bool pdl_waited = false;
    uint32_t tc0 = 0, tc1 = 0, te = 0;  // tiles so far, by stream and in all
    TItem it, nx;
    bool have = t_item(L, 0, it), ok = true;
    if (have) {
      t_load_requests(L.jobs[it.job], it, res0, warp - kTEpiWarp0, lane);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mb::arrive(&reqf);
    }
    for (uint32_t r = 0; ok && have; ++r) {
      const bool more = t_item(L, r + 1, nx);
      const TJob& J = L.jobs[it.job];
      const uint32_t N = J.mb_rows, c0 = N > 64 ? 64 * half : 32 * half;
      const bool two = N > 64 && c0 + 32 < N;  // this warp reads a second 32 columns
      // the next item's requests are announced once both issuers have seen this
      // item's (asked by one of the warps whose arrivals announce them, and here, while
      // the first counts are still to come)
      const bool seen = warp != kTEpiWarp0 || lane != 0 || !more ||
                        mb::wait(&reqe, r & 1u, abort_flag, status, kTWaitNs);
      uint32_t t = it.t0;
      for (uint32_t i = 0; i < it.nt; ++i, t += J.splits, ++te) {
        const uint32_t g = i % kTStreams, c = g ? tc1++ : tc0++, buf = nb2 & c;
        if (!mb::wait(&accf[g][buf], (c >> nb2) & 1u, abort_flag, status, kTWaitNs)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncwarp();
        uint32_t pw0, pw1 = 0;  // parities of this column, 32 requests a word
        const uint32_t acc = tmem + ((32u * quarter) << 16) + g * kTAcc + buf * kTAccHalf + c0;
        if constexpr (G == 1) {
          uint32_t r0[32], r1[32];
          t_ld32(acc, r0);  // (columns past N: not used)
          if (two) t_ld32(acc + 32, r1);
          t_wait_ld();
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mb::arrive(&acce[g][buf]);
          pw0 = t_parities(r0);
          if (two) pw1 = t_parities(r1);
        } else {  // (fewer registers a thread)
          uint32_t r0[32];
          t_ld32(acc, r0);
          t_wait_ld();
          if (two) {
            pw0 = t_parities(r0);
            t_ld32(acc + 32, r0);
            t_wait_ld();
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mb::arrive(&acce[g][buf]);
          if (two)
            pw1 = t_parities(r0);
          else
            pw0 = t_parities(r0);
        }
        if (more && i + 1 == it.nt) {
          // every tile's MMAs have read the item's requests: the next item's
          // go in before this tile's replies, so that its MMAs start the sooner
          t_load_requests(L.jobs[nx.job], nx, res0, warp - kTEpiWarp0, lane);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0 && seen) mb::arrive(&reqf);
        }
        const WarpTranspose transpose;  // formed anew for each tile: its registers are the counts' before
        const uint32_t ob = out0 + (te & 1u) * kTOutBytes, oq = ob + (c0 + lane) * 16u + quarter * 4u;
        if (c0 < N)
          asm volatile("st.shared.b32 [%0], %1;" ::"r"(oq), "r"(transpose(pw0)) : "memory");
        if (two)
          asm volatile("st.shared.b32 [%0], %1;" ::"r"(oq + 512u), "r"(transpose(pw1)) : "memory");
        __syncwarp();
        if (lane == 0) mb::arrive(&outf);
        if (!pdl_waited) {
          asm volatile("griddepcontrol.wait;" ::: "memory");  // replies initialised / released
          pdl_waited = true;
        }
        // two buffers: a thread writes one again only after this barrier's next
        // phase, which every thread joins with its reads of this one behind it
        if (!mb::wait(&outf, te & 1u, abort_flag, status, kTWaitNs)) {
          ok = false;
          break;
        }
        // two threads per request, eight bytes each
        const uint32_t q = et >> 1, b = it.b0 + q;
        if (q < N && b < J.B) {
          uint64_t v;
          asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(ob + et * 8u) : "memory");
          const uint32_t w = t * 4u + (et & 1u) * 2u;
          uint32_t* p = J.out + static_cast<uint64_t>(b) * J.Wd + w;
          if (J.split == 2) v ^= t_mask(J.seeds + static_cast<uint64_t>(b) * 32, w);
          if (J.split == 1)
            asm volatile("red.relaxed.gpu.global.xor.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
          else
            *reinterpret_cast<uint64_t*>(p) = v;
        }
      }
      it = nx;
      have = more;
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kTEpiWarp0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTTmemCols)
                 : "memory");
}

// Initialises the replies of the jobs that XOR-reduce into them (zeros, or
// the masks of a masked job) before the scan: grid.y = job.  PDL-chained like
// the scan, it waits for the previous kernel before writing.
template <int NJ>
__global__ void gf2_tmem_init_kernel(const __grid_constant__ TLaunch<NJ> L) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const TJob& J = L.jobs[blockIdx.y];
  if (J.split != 1) return;
  init_replies(reinterpret_cast<uint4*>(J.out), J.B, J.Wd / 4, J.seeds,
               blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, (uint64_t)gridDim.x * blockDim.x);
}

// Blocks of up to 112 requests take the layout with two expander groups.
int t_groups(uint32_t N) { return N <= TLayout<2>::kAcc ? 2 : 1; }
// Clocks of an item: W words (K = 64 steps, whole stages of four) of nt tiles at
// N requests, fitted to measured launches.  The two
// streams together run a step in 0.54 N clocks (the MMA) or 48 (instruction
// latency); one alone in 115, and it stands still while a tile's counts are read.
double t_item_clk(uint32_t N, uint32_t W, uint32_t nt) {
  const double steps = (W + 3) / 4 * 4;
  const double both = nt * (steps * std::max(0.54 * N, 48.0) + 40.0);
  const double one = ((nt + 1) / 2) * (steps * 115.0 + (N <= kTAccHalf ? 400.0 : 400.0 + 10.0 * N));
  return 6000.0 + 0.3 * N * W + std::max(both, one);
}

TJob t_job(const uint64_t* R, uint32_t words64, uint32_t B, uint32_t* out, const uint8_t* seeds,
           uint64_t n, uint32_t Wd) {
  TJob j{};
  j.R = R;
  j.out = out;
  j.seeds = seeds;
  j.n = n;
  j.Wd = Wd;
  j.words64 = words64;
  j.B = B;
  j.nw = static_cast<uint32_t>((n + 63) / 64);
  j.tiles = Wd / 4;
  j.mbs = (B + kTMaxN - 1) / kTMaxN;
  j.mb_rows = ((B + j.mbs - 1) / j.mbs + 15) / 16 * 16;
  return j;
}

uint32_t t_max_words(uint32_t N) { return (t_groups(N) == 2 ? TLayout<2>::kRes : TLayout<1>::kRes) / (32 * N); }

// How a job's replies are stored with kcs k-chunks (TJob::split).  A masked read of
// a table so small that every CTA has a tile at most forms the masks where it stores
// (a keystream block per eight bytes, but no launch before it: 90 masked reads of 1 132
// x 256 bytes 5.0 us, 6.8 with one); larger ones have them written first, a block
// per 64 bytes.
uint32_t t_split(const TJob& j, uint32_t kcs) {
  if (kcs > 1) return 1;
  if (!j.seeds) return 0;
  return static_cast<uint64_t>(j.mbs) * j.tiles <= static_cast<uint64_t>(device_sm_count()) ? 2 : 1;
}
// What that adds to a launch, in clocks: the replies' initialisation, or masks
// formed at the stores of `nt` tiles of an item.
double t_split_clk(const TJob& j, uint32_t kcs, uint32_t nt) {
  const uint32_t split = t_split(j, kcs);
  if (split == 0) return 0.0;
  if (split == 2) return 1800.0 * nt;
  return j.seeds && kcs > 1 ? 5000.0 : 3000.0;
}

void t_set_chunks(TJob& j, uint32_t kc_words, uint32_t splits) {
  j.kc_words = kc_words;
  j.kcs = (j.nw + kc_words - 1) / kc_words;
  j.splits = splits;
  j.split = t_split(j, j.kcs);
}

uint32_t t_min_chunks(const TJob& j) {
  const uint32_t maxw = t_max_words(j.mb_rows);
  return (j.nw + maxw - 1) / maxw;
}

// A launch of however little work: its words have to come, be expanded, multiplied
// and read back (2 500 x 256 bytes at 48 requests 5.5 us in one k-chunk, 7.2 with ten
// and their replies' initialisation, which the items' times alone made 4.9).
constexpr double kTLeastClk = 12500.0;

// k-chunks and column splits of a one-job launch: the least rounds x item
// time over the chunk counts from the fewest that fit on, or with chunks of
// `fixed` words (0: none given).  Returns the clocks.
double t_plan(TJob& j, uint32_t grid, uint32_t fixed = 0) {
  // the last plans of this thread, by what they depend on (the search takes the host
  // 1.3 us, a third of a small read)
  struct Plan {
    uint32_t nw = 0, tiles = 0, mbs = 0, N = 0, fixed = 0, grid = 0, kw = 0, s = 0;
    bool masked = false;
    double clk = 0.0;
  };
  static thread_local Plan plans[16];
  Plan& p = plans[(j.nw * 0x9E3779B1u ^ j.tiles * 0x85EBCA77u ^ (j.mbs * 128u + j.mb_rows) * 0xC2B2AE3Du) >> 28];
  if (p.nw == j.nw && p.tiles == j.tiles && p.mbs == j.mbs && p.N == j.mb_rows && p.fixed == fixed &&
      p.grid == grid && p.masked == (j.seeds != nullptr)) {
    t_set_chunks(j, p.kw, p.s);
    return p.clk;
  }
  const uint32_t c0 = t_min_chunks(j);
  double best = 1e300;
  uint32_t bw = 1, bs = 1;
  for (uint32_t c = c0; c <= std::min<uint32_t>(j.nw, c0 + 40); ++c) {
    const uint32_t kw = fixed ? fixed : (j.nw + c - 1) / c;
    const uint64_t per = static_cast<uint64_t>(j.mbs) * ((j.nw + kw - 1) / kw);
    for (uint32_t k = 1; k <= 4; ++k) {
      uint32_t s = static_cast<uint32_t>(std::min<uint64_t>(j.tiles, k * grid / per));
      if (s < 1) s = 1;
      const uint32_t st = (j.tiles + s - 1) / s;
      const uint64_t items = per * s;
      const uint64_t rounds = (items + grid - 1) / grid;
      const double cost = std::max(static_cast<double>(rounds) * t_item_clk(j.mb_rows, kw, st), kTLeastClk) +
                          t_split_clk(j, (j.nw + kw - 1) / kw, st);
      if (cost < best) {
        best = cost;
        bw = kw;
        bs = s;
      }
    }
    if (fixed) break;
  }
  t_set_chunks(j, bw, bs);
  p = Plan{j.nw, j.tiles, j.mbs, j.mb_rows, fixed, grid, bw, bs, j.seeds != nullptr, best};
  return best;
}

// The replies that a launch XOR-reduces into, initialised before it.  Masks take
// time: they are spread over the SMs in CTAs of 64 threads, one of which fits beside a
// CTA of the scan before it (G = 1).  Beside one of G = 2, which leaves no registers,
// none does: started early, they go to the first SMs that it leaves, four at most to
// each by the shared memory they ask for (48 masked reads of 32 768 x 4 KiB 37 us, 45
// in CTAs of 256 without, 39 when they wait for the scan's end).
template <int NJ>
cudaError_t t_init(const TLaunch<NJ>& L, int G, cudaStream_t st) {
  bool any = false;
  uint64_t blocks = 0;  // keystream blocks of the job with the most masks
  for (uint32_t i = 0; i < L.njobs; ++i) {
    if (L.jobs[i].split != 1) continue;
    any = true;
    if (L.jobs[i].seeds) blocks = std::max(blocks, static_cast<uint64_t>(L.jobs[i].B) * ((L.jobs[i].Wd + 15) / 16));
  }
  if (!any) return cudaSuccess;
  if (!blocks) return launch_pdl(gf2_tmem_init_kernel<NJ>, dim3(64, L.njobs), dim3(256), 0, st, L);
  const uint32_t ctas = static_cast<uint32_t>(std::min<uint64_t>((blocks + 63) / 64, 256));
  return launch_pdl(gf2_tmem_init_kernel<NJ>, dim3(ctas, L.njobs), dim3(64), G == 2 ? 48u * 1024u : 0u, st, L);
}

template <int NJ, int G>
cudaError_t t_scan(TLaunch<NJ>& L, cudaStream_t st) {
  using Y = TLayout<G>;
  static std::atomic<bool> ready{false};  // idempotent set-up: a race only repeats it
  if (!ready.load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(gf2_tmem_kernel<NJ, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, Y::kSmem);
    if (e != cudaSuccess) return e;
    ready.store(true, std::memory_order_release);
  }
  int* status = device_status_word();
  if (!status) return cudaErrorInvalidSymbol;
  // two accumulators per stream where every block's requests fit beside others
  L.nbuf = 2u;
  for (uint32_t i = 0; i < L.njobs; ++i)
    if (L.jobs[i].mb_rows > Y::kAcc - kTAccHalf) L.nbuf = 1u;
  const uint32_t grid = std::min<uint32_t>(L.total_items, device_sm_count());
  return launch_pdl(gf2_tmem_kernel<NJ, G>, dim3(grid), dim3(Y::kThreads), Y::kSmem, st, L, status);
}

}  // namespace

// (with a launch and, where masks are reduced into, their share of it that no chunking
// changes; 4 % more than fitted: where the two forms are as close as that, the other one is taken)
double gf2_tmem_clk(uint64_t n, uint32_t Wd, uint32_t B, bool masked) {
  static const uint8_t some = 0;  // (a masked job plans as one; nothing is read)
  TJob j = t_job(nullptr, 0, B, nullptr, masked ? &some : nullptr, n, Wd);
  const double clk = t_plan(j, static_cast<uint32_t>(device_sm_count()));
  return 1.04 * (clk + (masked && j.kcs > 1 ? 6000.0 : 1000.0));
}

uint32_t gf2_tmem_max_rows(uint32_t B) {
  return 64u * t_max_words(t_job(nullptr, 0, B, nullptr, nullptr, 64, 4).mb_rows);
}

cudaError_t launch_gf2_tmem(const uint64_t* Tt, uint64_t n, uint32_t Wd, const uint64_t* R,
                            uint32_t words64, uint32_t B, uint32_t* out, const uint8_t* seeds,
                            cudaStream_t st, uint32_t kc_rows) {
  if (B == 0) return cudaSuccess;
  TLaunch<1> L{};
  L.njobs = 1;
  TJob J = t_job(R, words64, B, out, seeds, n, Wd);
  const uint32_t grid = static_cast<uint32_t>(device_sm_count());
  t_plan(J, grid, kc_rows ? std::min(t_max_words(J.mb_rows), std::max<uint32_t>(1, kc_rows / 64)) : 0u);
  const uint64_t items = static_cast<uint64_t>(J.mbs) * J.kcs * J.splits;
  if (items > 0xFFFFFFFFull) return cudaErrorInvalidValue;
  L.total_items = static_cast<uint32_t>(items);
  L.jobs[0] = J;
  cudaError_t e = gf2_table_map(Tt, n, Wd, kTCols, &L.maps[0]);
  if (e != cudaSuccess) return e;
  e = t_init(L, t_groups(J.mb_rows), st);
  if (e != cudaSuccess) return e;
  return t_groups(J.mb_rows) == 2 ? t_scan<1, 2>(L, st) : t_scan<1, 1>(L, st);
}

// Up to kTMultiJobs jobs of one layout for one persistent launch: k-chunks as
// long as they fit, cut into column runs of about equal cost (six items per
// CTA: 2 156 us for 16 uneven tables, 2 275 with three, 2 160 with twelve), the
// jobs in descending item cost.
static cudaError_t t_build_multi(const M4Request* reqs, uint32_t count, TLaunch<kTMultiJobs>& L) {
  const uint32_t grid = static_cast<uint32_t>(device_sm_count());
  std::vector<TJob> js;
  std::vector<const M4Request*> src;
  double total = 0.0;
  for (uint32_t i = 0; i < count; ++i) {
    const M4Request& q = reqs[i];
    if (q.B == 0) continue;
    if (!q.Tt) return cudaErrorInvalidValue;
    TJob j = t_job(q.R, q.words64, q.B, q.out, q.seeds, q.n, q.Wd);
    const uint32_t c = t_min_chunks(j);
    t_set_chunks(j, (j.nw + c - 1) / c, 1);
    total += static_cast<double>(j.mbs) * j.kcs * t_item_clk(j.mb_rows, j.kc_words, j.tiles);
    js.push_back(j);
    src.push_back(&q);
  }
  const double target = total / (6.0 * grid);
  std::vector<double> cost(js.size());
  std::vector<size_t> order(js.size());
  for (size_t i = 0; i < js.size(); ++i) {
    TJob& j = js[i];
    const double whole = t_item_clk(j.mb_rows, j.kc_words, j.tiles);
    const uint32_t s = std::max<uint32_t>(1, std::min<uint32_t>((j.tiles + 1) / 2, static_cast<uint32_t>(whole / target + 0.5)));
    t_set_chunks(j, j.kc_words, s);
    cost[i] = t_item_clk(j.mb_rows, j.kc_words, (j.tiles + s - 1) / s);
    order[i] = i;
  }
  std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t b) { return cost[a] > cost[b]; });
  L.njobs = 0;
  uint64_t items = 0;
  for (size_t oi : order) {
    TJob j = js[oi];
    j.item_begin = static_cast<uint32_t>(items);
    items += static_cast<uint64_t>(j.mbs) * j.kcs * j.splits;
    if (items > 0xFFFFFFFFull) return cudaErrorInvalidValue;
    const cudaError_t e = gf2_table_map(src[oi]->Tt, j.n, j.Wd, kTCols, &L.maps[L.njobs]);
    if (e != cudaSuccess) return e;
    L.jobs[L.njobs++] = j;
  }
  L.total_items = static_cast<uint32_t>(items);
  return cudaSuccess;
}

cudaError_t launch_gf2_tmem_multi(const M4Request* reqs, uint32_t count, cudaStream_t st) {
  // The jobs of each layout in launches of their own (16 uneven tables 2 156 us
  // in one launch of the layout for larger blocks, 1 942 in two); every launch's
  // replies are initialised before the first scan, so that a scan's CTAs start
  // on the SMs that the scan before it leaves.
  std::vector<M4Request> part[2];
  for (uint32_t i = 0; i < count; ++i) {
    if (reqs[i].B == 0) continue;
    if (!reqs[i].Tt) return cudaErrorInvalidValue;
    const TJob j = t_job(reqs[i].R, reqs[i].words64, reqs[i].B, nullptr, nullptr, reqs[i].n, reqs[i].Wd);
    part[t_groups(j.mb_rows) - 1].push_back(reqs[i]);
  }
  std::vector<TLaunch<kTMultiJobs>> ls;
  std::vector<int> layout;
  for (int g = 0; g < 2; ++g)
    for (size_t i = 0; i < part[g].size(); i += kTMultiJobs) {
      ls.emplace_back();
      layout.push_back(g + 1);
      const cudaError_t e = t_build_multi(
          part[g].data() + i, static_cast<uint32_t>(std::min<size_t>(kTMultiJobs, part[g].size() - i)), ls.back());
      if (e != cudaSuccess) return e;
    }
  for (size_t i = 0; i < ls.size(); ++i) {
    const cudaError_t e = t_init(ls[i], layout[i], st);
    if (e != cudaSuccess) return e;
  }
  for (size_t i = 0; i < ls.size(); ++i) {
    const cudaError_t e = layout[i] == 2 ? t_scan<kTMultiJobs, 2>(ls[i], st) : t_scan<kTMultiJobs, 1>(ls[i], st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace tpir
