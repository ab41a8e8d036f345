// CTA-pair tensor-core form of the batched PIR read for more than 128
// requests (gf2tmem.cu holds the form for the rest and the choice's other
// side): the exact 0/1 integer product on tcgen05.mma kind::mxf4 with both
// operands in shared memory, accumulated in fp32 in tensor memory; an output
// bit is the parity of its count.
//
// Operands.  Both matrices are 4-bit e2m1 values (a set bit = 1.0, packed two
// per byte) in the block-scaled MMA (every scale factor 1.0 = UE8M0 0x7F):
// products are 0 or 1 and a k-chunk's counts stay <= 32 768, exact in fp32.
// Packed 4-bit operands are taken only K-major, so the table is read from its
// bit-transposed copy (tcopy.cu: for each column, 64 buckets' bits in one
// word), and the request rows are K-major by nature.  Both use one order of the
// buckets within a 32-bucket chunk: element 8 t + m of the chunk (nibble m of
// its 32-bit word t) is bucket 4 m + t, so a word's 32 bits become their 32
// nibbles with one shift and one mask per 8 nibbles.  Every wait is bounded; a
// wait that gives up sets the status word, and the CTA drains its MMAs and TMA
// loads and frees its tensor memory before it returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "chacha.cuh"
#include "mbar.cuh"
#include "tpir_internal.h"

namespace tpir {
namespace {

constexpr int kGKStage = 256;                    // buckets per stage
constexpr int kGStageWords = kGKStage / 64;      // 64-bit words of a request row / table column per stage
constexpr int kGKStep = 64;                      // buckets per MMA
constexpr int kGCols = 224;                      // table columns per strip (MMA N)
constexpr int kGStripWords = kGCols / 32;        // reply words per strip
constexpr int kGRowBytes = kGKStage / 2;         // operand bytes per row per stage (e2m1)
// K-major, no swizzle: 8-row x 16-byte core matrices, kGLbo apart along K,
// kGSbo apart along M / N.  Row r, byte k of an operand: (r / 8) kGSbo +
// (k / 16) kGLbo + (r % 8) 16.
constexpr int kGLbo = 128;
constexpr int kGSbo = (kGRowBytes / 16) * 128;
constexpr uint32_t kGTmaWarp = 0, kGEpiWarp0 = 16, kGIssueWarp = 24;
// Roles by SM sub-partition (warp w issues from sub-partition w % 4).  The
// MMA thread (warp 24) issues from sub-partition 0, and any expander placed
// there fell up to a pipeline stage behind the rest (its shared-memory
// traffic queued behind the tensor-core instructions) while every stage waits
// for its last expander.  So sub-partition 0 holds only the TMA producer (0),
// the epilogue warps 16 and 20 and the MMA thread; the expanders share
// sub-partitions 1-3.
__device__ __forceinline__ int g_table_index(uint32_t warp) {
  switch (warp) {
    case 1: return 0; case 5: return 1; case 9: return 2; case 13: return 3;
    case 3: return 4; case 7: return 5; case 11: return 6;
    default: return -1;
  }
}
constexpr uint32_t kGTmemCols = 512;
constexpr uint32_t kGSfCol = 448;                // scale factors: columns 448..511 (UE8M0 1.0)
constexpr uint32_t kGSfa = 448, kGSfb = 480;
constexpr uint64_t kGWaitNs = 4000000000ull;
constexpr uint64_t kGMaxCount = 32768;           // largest count one accumulator holds

// Descriptor increment of one K-step (two 16-byte chunks).
constexpr uint64_t kDescK = (2 * kGLbo) >> 4;

// One table's read in a launch (one job of a many-table launch).
struct GJob {
  const uint64_t* R;
  uint32_t* out;
  const uint8_t* seeds;  // masks of a serialized-PIR read, or null
  uint64_t n;
  uint32_t Wd, words64, B;
  uint32_t n_strips, n_mb, kc_rows;
  uint32_t split;        // 0: replies stored; 1: initialised first (zeros or masks)
                         // and XOR-reduced into; 2: masked, stored by their single
                         // writer (one k-chunk, items) with the mask XORed in
};

// A launch: the job with the tensor maps of its transposed table and of its
// request rows, in the kernel parameters.
struct GLaunch {
  CUtensorMap map;
  CUtensorMap rmap;    // request rows (RM 1) or even rows (RM 2) as 64-bit words
  CUtensorMap rmap_o;  // RM 2: row pairs as 64-bit words (odd rows' boxes)
  GJob job;
  uint32_t total_items;
};

// Shared-memory matrix descriptor, K-major without swizzle.
__device__ __forceinline__ uint64_t g_desc(uint32_t addr) {
  return static_cast<uint64_t>((addr >> 4) & 0x3FFFu) | (static_cast<uint64_t>(kGLbo >> 4) << 16) |
         (static_cast<uint64_t>(kGSbo >> 4) << 32) | (1ull << 46);
}

// byte offset of (row, 16-byte chunk) in an operand tile of a stage
__device__ __forceinline__ uint32_t g_off(uint32_t row, uint32_t chunk) {
  return (row >> 3) * kGSbo + chunk * kGLbo + (row & 7u) * 16u;
}

// 32 buckets' bits (bit i = bucket i of the chunk) as 32 e2m1 nibbles, 1.0
// (0x2) where set: nibble m of word t is bucket 4 m + t.
__device__ __forceinline__ uint4 g_spread(uint32_t h) {
  constexpr uint32_t m = 0x22222222u;
  return make_uint4((h << 1) & m, h & m, (h >> 1) & m, (h >> 2) & m);
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}

__device__ __forceinline__ uint64_t ld_shared_u64(uint32_t addr) {
  uint64_t v;
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// 2-D TMA load of a box at (x, y) into shared memory, completing its bytes
// on the mbarrier (whose expected transaction count the caller has raised)
__device__ __forceinline__ void g_tma_load(uint32_t dst, const CUtensorMap* map, int x, int y,
                                           uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(mb::saddr(bar))
      : "memory");
}

__device__ __forceinline__ void g_red_xor32(uint32_t* p, uint32_t v) {
  asm volatile("red.relaxed.gpu.global.xor.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void g_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Word i (0..15) of a keystream block, by selects (the index is not known at
// compile time; a register array indexed at run time would go to local memory)
__device__ __forceinline__ uint32_t g_pick(const uint32_t (&k)[16], uint32_t i) {
  uint32_t v = k[0];
#pragma unroll
  for (uint32_t j = 1; j < 16; ++j) v = i == j ? k[j] : v;
  return v;
}

// Parity words of `nw` (<= 7) consecutive reply words (w0 ..) for request b
// from the accumulator columns at taddr (column 32 c + j = bit j of word
// w0 + c): each value is an exact count; adding 2^23 puts it in the
// mantissa, whose lowest bit is the count's parity.  Written, or XOR-reduced
// for a split k range or masked replies, into the reply row.
__device__ __forceinline__ void g_epilogue(const GJob& J, uint32_t taddr, uint32_t b, uint32_t w0,
                                           uint32_t nw) {
  uint32_t pw[kGStripWords];
#pragma unroll
  for (uint32_t c = 0; c < kGStripWords; ++c) {
    pw[c] = 0u;
    if (c < nw && w0 + c < J.Wd) {  // uniform across the warp
      uint32_t v[32];
      g_ld32(taddr + 32u * c, v);
      uint32_t w = 0;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        w |= (__float_as_uint(__uint_as_float(v[j]) + 8388608.0f) & 1u) << j;
      pw[c] = w;
    }
  }
  if (b >= J.B) return;
  uint32_t* o = J.out + static_cast<uint64_t>(b) * J.Wd + w0;
  if (J.split == 2) {
    // a masked reply word with this thread its only writer: XOR in the
    // request's keystream (ChaCha20 block w / 16, word w % 16; the seven words
    // span at most two blocks)
    const uint4* k4 = reinterpret_cast<const uint4*>(J.seeds + static_cast<uint64_t>(b) * 32);
    const uint4 ka = __ldg(k4), kb = __ldg(k4 + 1);
    const uint32_t key[8] = {ka.x, ka.y, ka.z, ka.w, kb.x, kb.y, kb.z, kb.w};
    const uint32_t blk0 = w0 >> 4;
    uint32_t k0[16], k1[16];
    cc_block(key, blk0, k0);
    cc_block(key, blk0 + 1, k1);
#pragma unroll
    for (uint32_t c = 0; c < kGStripWords; ++c) {
      const uint32_t w = w0 + c;
      const uint32_t m = (w >> 4) == blk0 ? g_pick(k0, w & 15u) : g_pick(k1, w & 15u);
      pw[c] ^= m;
    }
  }
#pragma unroll
  for (uint32_t c = 0; c < kGStripWords; ++c) {
    if (c < nw && w0 + c < J.Wd) {
      if (J.split == 1)
        g_red_xor32(o + c, pw[c]);
      else
        o[c] = pw[c];
    }
  }
}

// ---------------------------------------------------------------------------
// The CTA-pair form (tcgen05 cta_group::2), for one job of more than 128
// requests.  Two CTAs of a cluster share every MMA: M = 256 requests (128 in
// each CTA's shared memory) x N = 224 table columns (112 in each CTA's) x K =
// 64, issued by the even CTA, each CTA's tensor memory holding its 128
// requests' counts.  A pair item is (two strips = 448 columns, a block of up
// to 256 requests, a k-chunk): per stage each CTA expands its 128 request
// rows and 2 x 112 table columns (44 KiB, against 60 KiB for the 256 x 224 of
// a single CTA) and each MMA reads 7.5 KiB of its shared memory (against 11
// KiB): the shared-memory traffic per multiply-add that bounds the kernel
// falls by about 30 %.
//
// Per CTA: warp 0 TMA (the CTA's own raw stages), 7 table expanders (warps
// 1, 5, 9, 13, 3, 7, 11: lane = column 32 i + lane of the CTA's 224, i.e.
// tile c / 112, column c % 112 of that tile), 4 request expanders (warps 2,
// 6, 10, 14: lane = request 32 i + lane of the CTA's 128), the MMA thread
// (warp 24, even CTA only), 8 epilogue warps (16..23: N-tile (w - 16) / 4,
// lanes 32 (w % 4) ..), warps 4, 8, 12, 15 of the odd CTA relays (idle in
// the even one).  Every expander warp arrives at its own CTA's "full" barrier
// of the stage; in the odd CTA relay k (one thread) waits for the barriers of
// ring slot k and passes one cluster-scope arrival to the even CTA's "pfull"
// (such an arrival stalls its thread for hundreds of cycles: per expander warp
// it cost each warp about a thousand cycles a stage, and one relay thread for
// all slots fell behind), and the MMA thread waits for both.  The MMAs' commits arrive at the "empty"
// barriers of both CTAs (multicast), their accumulators' at both "accf"
// barriers; every epilogue warp of both arrives at the even CTA's "acce".
// All waits bounded; both CTAs meet at a cluster barrier before the tensor
// memory is freed.
constexpr int kPCols = 112;                          // table columns per CTA per N-tile
constexpr int kPTileA = 128 * kGRowBytes;            // 16 KiB: the CTA's 128 request rows
constexpr int kPTileB = kPCols * kGRowBytes;         // 14 KiB
constexpr int kPStageBytes = kPTileA + 2 * kPTileB;  // 44 KiB
constexpr int kPStages = 4;
constexpr int kPRaw = 4;
constexpr int kPRawTile = kPCols * kGStageWords * 8;  // 3.5 KiB: a tile's words of a stage
constexpr int kPRawTable = 2 * kPRawTile;
template <int RM>
__host__ __device__ constexpr int p_raw_req() { return RM == 1 ? 128 * 32 : 64 * 32 + 64 * 48; }
template <int RM>
__host__ __device__ constexpr int p_raw_bytes() { return kPRawTable + p_raw_req<RM>(); }
template <int RM>
__host__ __device__ constexpr int p_smem() { return 1024 + kPStages * kPStageBytes + kPRaw * p_raw_bytes<RM>(); }
static_assert(p_smem<1>() <= 231424 && p_smem<2>() <= 231424,
              "dynamic shared memory above 227 KiB less the static part");
constexpr uint32_t kPTableWarps = 7, kPReqWarps = 4;
constexpr int kPThreads = 25 * 32;
constexpr uint64_t kPDescStage = kPStageBytes >> 4;
constexpr uint64_t kPDescTileB = kPTileB >> 4;
// M = 256 (bits 24..28 = M / 16), N = 224, e2m1 x e2m1, UE8M0 scales
constexpr uint32_t kPIdesc = (1u << 7) | (1u << 10) | ((uint32_t)(kGCols >> 3) << 17) | (1u << 23) |
                             ((256u >> 4) << 24);

__device__ __forceinline__ int p_relay_index(uint32_t warp) {
  switch (warp) {
    case 4: return 0; case 8: return 1; case 12: return 2; case 15: return 3;
    default: return -1;
  }
}
static_assert(kPStages == 4, "one relay warp per ring slot");
__device__ __forceinline__ int p_req_index(uint32_t warp) {
  switch (warp) {
    case 2: return 0; case 6: return 1; case 10: return 2; case 14: return 3;
    default: return -1;
  }
}

__device__ __forceinline__ void p_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t sfa,
                                      uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%4], [%5], "
      "p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(kPIdesc), "r"(sfa), "r"(sfb), "r"(accumulate)
      : "memory");
}
// commit of the MMAs issued so far to the barrier at this offset in both CTAs
__device__ __forceinline__ void p_commit_both(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], "
      "%1;" ::"r"(mb::saddr(bar)),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}
__device__ __forceinline__ void p_commit_self(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   mb::saddr(bar))
               : "memory");
}

// Pair items: (pair strip, M-block, k-chunk), pair strip fastest; the pairs
// take them round by round, sweeping the grid in alternate directions.
struct PItem {
  uint32_t pstrip, b0;
  uint64_t k0, k1;
};
__device__ __forceinline__ bool p_item(const GLaunch& L, uint32_t pair, uint32_t npairs, uint32_t r,
                                       PItem& it) {
  const uint32_t c = (r & 1u) ? npairs - 1u - pair : pair;
  const uint32_t item = c + r * npairs;
  if (item >= L.total_items) return false;
  const GJob& J = L.job;
  const uint32_t nps = (J.n_strips + 1) / 2;
  it.pstrip = item % nps;
  const uint32_t rest = item / nps;
  it.b0 = (rest % J.n_mb) * 256u;
  it.k0 = static_cast<uint64_t>(rest / J.n_mb) * J.kc_rows;
  it.k1 = min(J.n, it.k0 + J.kc_rows);
  return true;
}
struct PCursor {
  uint32_t r;
  uint64_t ks;
  PItem it;
  bool valid;
};
__device__ __forceinline__ void p_cur_item(PCursor& c, const GLaunch& L, uint32_t pair, uint32_t npairs) {
  c.valid = p_item(L, pair, npairs, c.r++, c.it);
  if (c.valid) c.ks = c.it.k0;
}
__device__ __forceinline__ void p_cur_next(PCursor& c, const GLaunch& L, uint32_t pair, uint32_t npairs) {
  c.ks += kGKStage;
  if (c.ks >= c.it.k1) p_cur_item(c, L, pair, npairs);
}

template <int RM>
__global__ void __launch_bounds__(kPThreads, 1)
    gf2_mma_pair_kernel(const __grid_constant__ GLaunch L, int* status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kPStages], pfull[kPStages], empty[kPStages], accf, acce, drain;
  __shared__ __align__(8) uint64_t raw_full[kPRaw], raw_empty[kPRaw];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  uint8_t* stages = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t stage0 = mb::saddr(stages);
  const uint32_t raw0 = stage0 + kPStages * kPStageBytes;
  volatile int* abort_flag = &s_abort;
  constexpr int kRawBytes = p_raw_bytes<RM>();
  const uint32_t rank = mb::cluster_rank();
  const uint32_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kPStages; ++s) {
      mb::init(&full[s], kPTableWarps + kPReqWarps);  // this CTA's expander warps
      mb::init(&pfull[s], 1);                         // even CTA: the odd CTA's relay
      mb::init(&empty[s], 1);
    }
    mb::init(&accf, 1);
    mb::init(&acce, 2 * 8);  // every epilogue warp of both CTAs
    mb::init(&drain, 1);
    for (int s = 0; s < kPRaw; ++s) {
      mb::init(&raw_full[s], 1);
      mb::init(&raw_empty[s], kPTableWarps + kPReqWarps);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kGEpiWarp0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     mb::saddr(&s_tmem)),
                 "r"(kGTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  mb::cluster_sync();  // both CTAs' barriers initialised, tensor memory allocated
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  if (warp >= kGEpiWarp0 && warp < kGEpiWarp0 + 4) {
    const uint32_t one = 0x7F7F7F7Fu;  // scale factors 1.0, columns 448..511
    for (uint32_t col = kGSfCol; col < kGTmemCols; col += 8)
      asm volatile(
          "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(
              tmem + (((warp & 3u) * 32u) << 16) + col),
          "r"(one)
          : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  mb::cluster_sync();  // both CTAs' scale factors in place before the first MMA
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t lead_pfull0 = mb::cluster_addr(&pfull[0], 0);
  const uint32_t lead_acce = mb::cluster_addr(&acce, 0);

  if (warp == kGTmaWarp) {
    // ------------- this CTA's transposed-table words and request words -------------
    if (lane == 0) {
      uint32_t p = 0;
      PCursor c{};
      p_cur_item(c, L, pair, npairs);
      for (; c.valid; p_cur_next(c, L, pair, npairs), ++p) {
        const uint32_t rs = p % kPRaw, ph = (p / kPRaw) & 1u;
        if (!mb::wait_sleep(&raw_empty[rs], ph ^ 1u, abort_flag, status, kGWaitNs, 32)) break;
        const uint32_t dst = raw0 + rs * kRawBytes;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                         mb::saddr(&raw_full[rs])),
                     "r"(kRawBytes)
                     : "memory");
        const int kb = static_cast<int>(c.ks >> 6);
        const int x0 = static_cast<int>(c.it.pstrip * 2u * kGCols + rank * kPCols);
        g_tma_load(dst, &L.map, x0, kb, &raw_full[rs]);
        g_tma_load(dst + kPRawTile, &L.map, x0 + kGCols, kb, &raw_full[rs]);
        const int b = static_cast<int>(c.it.b0 + 128u * rank);
        if constexpr (RM == 1) {
          g_tma_load(dst + kPRawTable, &L.rmap, kb, b, &raw_full[rs]);
        } else {
          g_tma_load(dst + kPRawTable, &L.rmap, kb, b >> 1, &raw_full[rs]);
          g_tma_load(dst + kPRawTable + 64 * 32, &L.rmap_o,
                     static_cast<int>(L.job.words64) + kb - 1, b >> 1, &raw_full[rs]);
        }
      }
      for (uint32_t rs = 0; rs < static_cast<uint32_t>(kPRaw) && rs < p; ++rs) {
        const uint32_t last = rs + kPRaw * ((p - 1 - rs) / kPRaw);
        const uint64_t t0 = mb::gtimer();
        while (!mb::try_wait(&raw_full[rs], (last / kPRaw) & 1u)) {
          if (mb::gtimer() - t0 > kGWaitNs) {
            atomicExch(status, static_cast<int>(TPIR_ETIMEDOUT));
            break;
          }
        }
      }
    }
  } else if (g_table_index(warp) >= 0 || p_req_index(warp) >= 0) {
    // ------------------------------ expanders ------------------------------
    const bool table = g_table_index(warp) >= 0;
    const uint32_t idx = static_cast<uint32_t>(table ? g_table_index(warp) : p_req_index(warp));
    const uint32_t e = 32u * idx + lane;  // table column e of the CTA's 224, or request e of its 128
    const uint32_t t = e >= static_cast<uint32_t>(kPCols) ? 1u : 0u, cc = e - t * kPCols;
    uint32_t iter = 0;
    PCursor c{};
    p_cur_item(c, L, pair, npairs);
    for (; c.valid; p_cur_next(c, L, pair, npairs), ++iter) {
      const uint32_t rs = iter % kPRaw, rph = (iter / kPRaw) & 1u;
      const uint32_t s = iter % kPStages, ph = (iter / kPStages) & 1u;
      if (!mb::wait(&raw_full[rs], rph, abort_flag, status, kGWaitNs)) break;
      const uint32_t base = raw0 + rs * kRawBytes;
      uint64_t x[kGStageWords];
      if (table) {
#pragma unroll
        for (int i = 0; i < kGStageWords; ++i)
          x[i] = ld_shared_u64(base + t * kPRawTile + i * (kPCols * 8) + cc * 8u);
      } else if constexpr (RM == 1) {
        const uint32_t a = base + kPRawTable + e * 32u, h = (e >> 2) & 1u;
        const uint4 v0 = ld_shared_v4(a + 16u * h), v1 = ld_shared_v4(a + 16u * (h ^ 1u));
        const uint4 lo = h ? v1 : v0, hi = h ? v0 : v1;
        x[0] = lo.x | static_cast<uint64_t>(lo.y) << 32;
        x[1] = lo.z | static_cast<uint64_t>(lo.w) << 32;
        x[2] = hi.x | static_cast<uint64_t>(hi.y) << 32;
        x[3] = hi.z | static_cast<uint64_t>(hi.w) << 32;
      } else {
        const uint32_t pr = e >> 1;
        const uint32_t a = (e & 1u) ? base + kPRawTable + 64u * 32u + pr * 48u + 8u
                                    : base + kPRawTable + pr * 32u;
#pragma unroll
        for (uint32_t i = 0; i < kGStageWords; ++i) x[i] = ld_shared_u64(a + 8u * i);
      }
      {
        uint32_t used = 0;
#pragma unroll
        for (int i = 0; i < kGStageWords; ++i)
          used ^= static_cast<uint32_t>(x[i]) ^ static_cast<uint32_t>(x[i] >> 32);
        asm volatile("fence.proxy.async.shared::cta;" ::"r"(used) : "memory");
        __syncwarp();
        if (lane == 0) mb::arrive(&raw_empty[rs]);
      }
      if (!mb::wait(&empty[s], ph ^ 1u, abort_flag, status, kGWaitNs)) break;
      const bool store = table || c.it.b0 + 128u * rank + e < L.job.B;
      if (store) {
        const uint32_t o = table ? stage0 + s * kPStageBytes + kPTileA + t * kPTileB + g_off(cc, 0)
                                 : stage0 + s * kPStageBytes + g_off(e, 0);
#pragma unroll
        for (int i = 0; i < kGStageWords; ++i) {
          st_shared_v4(o + (2 * i) * kGLbo, g_spread(static_cast<uint32_t>(x[i])));
          st_shared_v4(o + (2 * i + 1) * kGLbo, g_spread(static_cast<uint32_t>(x[i] >> 32)));
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mb::arrive(&full[s]);
    }
  } else if (rank == 1 && p_relay_index(warp) >= 0) {
    // ---- relays: the odd CTA's stages of ring slot k, one cluster-scope arrival each ----
    if (lane == 0) {
      const uint32_t k = static_cast<uint32_t>(p_relay_index(warp));
      uint32_t iter = 0;
      PCursor c{};
      p_cur_item(c, L, pair, npairs);
      for (; c.valid; p_cur_next(c, L, pair, npairs), ++iter) {
        if (iter % kPStages != k) continue;
        const uint32_t ph = (iter / kPStages) & 1u;
        if (!mb::wait(&full[k], ph, abort_flag, status, kGWaitNs)) break;
        mb::arrive_cluster(lead_pfull0 + 8u * k);
      }
    }
  } else if (warp == kGIssueWarp && rank == 0) {
    // ---------------------- MMA issue for the pair (one thread) ----------------------
    if (lane == 0) {
      const uint64_t adesc0 = g_desc(stage0), bdesc0 = g_desc(stage0 + kPTileA);
      const uint32_t sfa = tmem + kGSfa, sfb = tmem + kGSfb;
      uint32_t is = 0, iph = 0;
      for (uint32_t r = 0;; ++r) {
        PItem it;
        if (*abort_flag || !p_item(L, pair, npairs, r, it)) break;
        bool ok = true;
        if (r >= 1) ok = mb::wait_cluster(&acce, (r - 1u) & 1u, abort_flag, status, kGWaitNs);
        bool have = ok && mb::wait(&full[is], iph, abort_flag, status, kGWaitNs) &&
                    mb::wait_cluster(&pfull[is], iph, abort_flag, status, kGWaitNs);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        ok = have;
        for (uint64_t ks = it.k0; have; ks += kGKStage) {
          const uint32_t s = is;
          if (++is == kPStages) {
            is = 0;
            iph ^= 1u;
          }
          const bool more = ks + kGKStage < it.k1;
          const uint64_t sa = adesc0 + s * kPDescStage, sb = bdesc0 + s * kPDescStage;
          const uint32_t acc0 = ks > it.k0 ? 1u : 0u;
          const uint64_t left = it.k1 - ks;
          const uint32_t nk =
              left >= kGKStage ? 4u : static_cast<uint32_t>((left + kGKStep - 1) / kGKStep);
          for (uint32_t j = 0; j < nk; ++j)
#pragma unroll
            for (uint32_t t = 0; t < 2; ++t)
              p_mma(tmem + kGCols * t, sa + kDescK * j, sb + kPDescTileB * t + kDescK * j, sfa, sfb,
                    j ? 1u : acc0);
          p_commit_both(&empty[s]);
          if (!more) break;
          if (!mb::wait(&full[is], iph, abort_flag, status, kGWaitNs) ||
              !mb::wait_cluster(&pfull[is], iph, abort_flag, status, kGWaitNs)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        if (!ok) break;
        p_commit_both(&accf);
      }
      p_commit_self(&drain);
      const uint64_t t0 = mb::gtimer();
      while (!mb::try_wait(&drain, 0)) {
        if (mb::gtimer() - t0 > kGWaitNs) {
          atomicExch(status, static_cast<int>(TPIR_ETIMEDOUT));
          break;
        }
      }
    }
  } else if (warp >= kGEpiWarp0 && warp < kGEpiWarp0 + 8) {
    // ---------------- epilogue: this CTA's 128 requests x the item's 2 strips ----------------
    const uint32_t quarter = warp & 3u, half = (warp - kGEpiWarp0) >> 2;
    bool pdl_waited = false;
    for (uint32_t r = 0;; ++r) {
      PItem it;
      if (*abort_flag || !p_item(L, pair, npairs, r, it)) break;
      if (!mb::wait_sleep(&accf, r & 1u, abort_flag, status, kGWaitNs, 256)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!pdl_waited) {
        asm volatile("griddepcontrol.wait;" ::: "memory");  // replies initialised / released
        pdl_waited = true;
      }
      const uint32_t lanes = (32u * quarter) << 16;
      g_epilogue(L.job, tmem + lanes + kGCols * half,
                 it.b0 + 128u * rank + 32u * quarter + lane,
                 (2u * it.pstrip + half) * kGStripWords, kGStripWords);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mb::arrive_cluster(lead_acce);
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  mb::cluster_sync();  // the pair's MMAs are complete before either CTA frees its memory
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kGEpiWarp0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kGTmemCols)
                 : "memory");
}

PFN_cuTensorMapEncodeTiled_v12000 g_encoder() {
  static std::mutex mu;
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  std::lock_guard<std::mutex> g(mu);
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e == cudaSuccess && q == cudaDriverEntryPointSuccess && fn)
      encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  return encode;
}

// Tensor map of a transposed table as a 2-D array of 64-bit words (row_bits
// columns x ceil(n / 64) blocks), box `width` columns (224, or 112 for a CTA
// of a pair) x 4 blocks; encoded once per (copy, shape, box).
}  // namespace
cudaError_t gf2_table_map(const uint64_t* Tt, uint64_t n, uint32_t Wd, uint32_t width,
                          CUtensorMap* out) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, uint64_t, uint32_t, uint32_t>, CUtensorMap> cache;
  PFN_cuTensorMapEncodeTiled_v12000 encode = g_encoder();
  if (!encode) return cudaErrorNotSupported;
  std::lock_guard<std::mutex> g(mu);
  const auto key = std::make_tuple(static_cast<const void*>(Tt), n, Wd, width);
  const auto it = cache.find(key);
  if (it != cache.end()) {
    *out = it->second;
    return cudaSuccess;
  }
  CUtensorMap m;
  const uint64_t row_bits = static_cast<uint64_t>(Wd) * 32;
  const cuuint64_t dims[2] = {row_bits, (n + 63) / 64};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(row_bits) * 8};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(width), static_cast<cuuint32_t>(kGStageWords)};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<uint64_t*>(Tt), dims,
                            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  if (cache.size() > 4096) cache.clear();
  cache[key] = m;
  *out = m;
  return cudaSuccess;
}

namespace {
// Tensor map of request words as a 2-D array of 64-bit words: dims x by y
// rows stride_words apart, box bx words x by rows (zero fill outside).
cudaError_t g_req_map(const uint64_t* R, uint64_t x, uint64_t y, uint64_t stride_words, uint32_t bx,
                      uint32_t by, CUtensorMap* out) {
  PFN_cuTensorMapEncodeTiled_v12000 encode = g_encoder();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {x, y};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(stride_words) * 8};
  const cuuint32_t box[2] = {bx, by};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(out, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<uint64_t*>(R), dims,
                            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Job fields that do not depend on the k-chunking.
GJob g_job(const uint64_t* R, uint32_t words64, uint32_t B, uint32_t* out, const uint8_t* seeds,
           uint64_t n, uint32_t Wd) {
  GJob j{};
  j.R = R;
  j.out = out;
  j.seeds = seeds;
  j.n = n;
  j.Wd = Wd;
  j.words64 = words64;
  j.B = B;
  j.n_strips = (Wd + kGStripWords - 1) / kGStripWords;
  j.n_mb = (B + 255) / 256;
  return j;
}

// How TMA can stage a job's request words (0: it cannot, per-thread loads).
// TMA boxes start 16-byte aligned: the x coordinate of a stage's first word
// is a multiple of 4, so with R 16-byte aligned rows of an even number of
// words are staged as rows (1: box 4 words x min(B, 256) rows at (word,
// request)); rows of an odd number of words as row pairs, 16-byte aligned
// (2): the even rows' four words (x = word, pair rows of 2 words64 words, dims
// nw x ceil(B/2)), the odd rows' from the even word before theirs (x =
// words64 + word - 1 in the pair, box 6 words, dims words64 + nw x
// floor(B/2)), where nw = ceil(n/64) are the job's own words of a row: no box
// reads past them.
uint32_t g_req_mode(const uint64_t* R, uint32_t words64) {
  if (reinterpret_cast<uintptr_t>(R) & 15u) return 0;
  return (words64 & 1u) ? 2u : 1u;
}
// k-chunks of kc_rows buckets: a multiple of a stage, at most kGMaxCount (a
// k-chunk's counts stay within the range the fp32 accumulators hold exactly)
uint32_t g_clamp_rows(uint64_t rows, uint64_t n) {
  rows = std::max<uint64_t>(rows, kGKStage);
  rows = (rows + kGKStage - 1) / kGKStage * kGKStage;
  rows = std::min<uint64_t>(rows, (n + kGKStage - 1) / kGKStage * kGKStage);
  return static_cast<uint32_t>(std::min<uint64_t>(rows, kGMaxCount));
}

// Pairs a launch of the pair kernel can hold resident at once (clusters of
// two CTAs of one SM each), once per request-staging mode.
template <int RM>
int p_max_pairs() {
  static std::atomic<int> cached{0};
  int v = cached.load(std::memory_order_acquire);
  if (v) return v;
  cudaError_t e = cudaFuncSetAttribute(gf2_mma_pair_kernel<RM>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, p_smem<RM>());
  if (e != cudaSuccess) return -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(device_sm_count() & ~1));
  cfg.blockDim = dim3(kPThreads);
  cfg.dynamicSmemBytes = p_smem<RM>();
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  e = cudaOccupancyMaxActiveClusters(&clusters, gf2_mma_pair_kernel<RM>, &cfg);
  if (e != cudaSuccess || clusters <= 0) return -1;
  cached.store(clusters, std::memory_order_release);
  return clusters;
}

// Clocks of the pair form on the whole device, launch included, and its
// k-chunk rows (rounds x item time, about 119 cycles per pair MMA, two per
// K-step; the measured launches took 1.21 times that and 5 us: 83 us for 64 at
// 256 requests of 32 768 x 4 KiB, 10.8 for 3.5 at 1 024 x 4 KiB).
double g_pair_plan(uint64_t n, uint32_t Wd, uint32_t B, int pairs, uint32_t* kc_rows) {
  const GJob J = g_job(nullptr, 0, B, nullptr, nullptr, n, Wd);
  const uint64_t nps = (J.n_strips + 1) / 2;
  const uint64_t max_kc = std::max<uint64_t>(1, (n + kGKStage - 1) / kGKStage);
  const uint64_t min_kc = (n + kGMaxCount - 1) / kGMaxCount;
  double best = 1e300;
  for (uint64_t c = std::max<uint64_t>(1, min_kc);
       c <= std::max<uint64_t>(min_kc, std::min<uint64_t>(max_kc, 512)); ++c) {
    const uint64_t rows = g_clamp_rows((n + c - 1) / c, n);
    const uint64_t kcs = (n + rows - 1) / rows;
    const uint64_t items = nps * J.n_mb * kcs;
    const uint64_t rounds = (items + pairs - 1) / pairs;
    const double cost = static_cast<double>(rounds) *
                        (static_cast<double>(rows) / kGKStep * 2.0 * 119.0 + 3000.0);
    if (cost < best) {
      best = cost;
      *kc_rows = static_cast<uint32_t>(rows);
    }
  }
  return 1.21 * best + 10000.0;
}

// One job on CTA pairs (B > 128, request rows TMA-staged): items of whole
// k-chunks taken round by round, k-chunks chosen like the single-CTA item
// schedule (about 119 cycles per pair MMA, two per K-step).
template <int RM>
cudaError_t g_launch_pair(const uint64_t* Tt, uint64_t n, uint32_t Wd, const uint64_t* R,
                          uint32_t words64, uint32_t B, uint32_t* out, const uint8_t* seeds,
                          cudaStream_t st, const GSched* sched) {
  const int pairs = p_max_pairs<RM>();
  if (pairs <= 0) return cudaErrorNotSupported;
  int* status = device_status_word();
  if (!status) return cudaErrorInvalidSymbol;
  GLaunch L{};
  GJob J = g_job(R, words64, B, out, seeds, n, Wd);
  const uint64_t nps = (J.n_strips + 1) / 2;
  g_pair_plan(n, Wd, B, pairs, &J.kc_rows);
  if (sched && sched->mode == 2 && sched->kc_rows) J.kc_rows = g_clamp_rows(sched->kc_rows, n);
  const uint64_t kcs = (n + J.kc_rows - 1) / J.kc_rows;
  const uint64_t items = nps * J.n_mb * kcs;
  if (items > 0xFFFFFFFFull) return cudaErrorInvalidValue;
  J.split = kcs > 1 ? 1u : seeds ? 2u : 0u;
  const uint64_t nw = (n + 63) / 64;
  if (RM == 1) {
    if (g_req_map(R, nw, B, words64, kGStageWords, 128, &L.rmap) != cudaSuccess)
      return cudaErrorInvalidValue;
  } else {
    if (g_req_map(R, nw, (B + 1) / 2, 2ull * words64, kGStageWords, 64, &L.rmap) != cudaSuccess ||
        g_req_map(R, words64 + nw, B / 2, 2ull * words64, kGStageWords + 2, 64, &L.rmap_o) !=
            cudaSuccess)
      return cudaErrorInvalidValue;
  }
  L.job = J;
  L.total_items = static_cast<uint32_t>(items);
  cudaError_t e = gf2_table_map(Tt, n, Wd, kPCols, &L.map);
  if (e != cudaSuccess) return e;
  // (masks in CTAs of 64 threads, some of which fit beside a CTA of the scan before)
  if (J.split == 1) e = launch_init_replies(reinterpret_cast<uint4*>(out), B, Wd / 4, seeds, st, 64);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * std::min<uint64_t>(items, pairs)));
  cfg.blockDim = dim3(kPThreads);
  cfg.dynamicSmemBytes = p_smem<RM>();
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, gf2_mma_pair_kernel<RM>, L, status);
  if (e == cudaSuccess) count_launches();
  return e;
}

}  // namespace

cudaError_t launch_gf2_mma(const uint64_t* Tt, uint64_t n, uint32_t Wd, const uint64_t* R,
                           uint32_t words64, uint32_t B, uint32_t* out, const uint8_t* seeds,
                           cudaStream_t st, const GSched* sched) {
  if (B == 0) return cudaSuccess;
  // CTA pairs take reads of more than one M-tile of requests whose rows TMA can
  // stage, where they are estimated (or were tuned) to be the faster form; a
  // device that cannot hold their clusters takes the other form.
  const uint32_t mode = sched ? (sched->loads ? 1u : sched->mode) : 0u;
  const uint32_t rm = B > 128 && (mode == 0 || mode == 2) ? g_req_mode(R, words64) : 0u;
  if (rm) {
    const int pairs = rm == 1 ? p_max_pairs<1>() : p_max_pairs<2>();
    uint32_t rows = 0;
    bool pair = pairs > 0 && mode == 2;
    if (pairs > 0 && mode == 0) {
      // (masks take 1.4 to 7 us, formed where a single k-chunk's replies are stored or
      // written before the scan)
      const double clk = g_pair_plan(n, Wd, B, pairs, &rows) + (seeds ? 7000.0 : 0.0);
      pair = clk < gf2_tmem_clk(n, Wd, B, seeds != nullptr);
    }
    if (pair)
      return rm == 1 ? g_launch_pair<1>(Tt, n, Wd, R, words64, B, out, seeds, st, sched)
                     : g_launch_pair<2>(Tt, n, Wd, R, words64, B, out, seeds, st, sched);
  }
  return launch_gf2_tmem(Tt, n, Wd, R, words64, B, out, seeds, st, sched ? sched->kc_rows : 0u);
}

}  // namespace tpir
