// Bit-transposed copy of a table for the tensor-core read.
//
// The tensor-core kernel multiplies the request bits by the table bits with
// packed 4-bit operands, which the tensor cores accept only K-major: for each
// table column (bit c of a row), its bits over consecutive buckets must be
// contiguous.  The row-major table (a bucket's row contiguous) is therefore
// kept a second time, bit-transposed in 64-bucket blocks:
//
//   Tt[kb][c]  (uint64)  bit i = bit c of the row of bucket 64 kb + i
//                        (bit c of a row: bit c % 8 of byte c / 8, LSB first);
//                        buckets past n are zero.
//
// The copy is built in full on first use and after a bulk load, and block by
// block after the slot moves of a write (only the moved slots' columns of the
// 64-bucket blocks holding them), in the same stream order as the table itself, so it always
// matches the table for every later read.
#include <algorithm>
#include <vector>

#include "bits.cuh"
#include "tpir_internal.h"

namespace tpir {
namespace {

// One work item: block kb (64 buckets) x 32 words of the row.  The 64 x 128
// bytes come in by whole 128-byte lines, and with COPY go out to the table (a
// bulk load from device memory: the source is read once for both); each warp
// then takes four words: lane l holds word w of buckets 64 kb + l and 64 kb +
// 32 + l, and two 32 x 32 transposes in registers give lane j column 32 w + j
// over the 64 buckets (32 lanes x 8 bytes stored, contiguous).
// Bound by HBM: a load of 32 768 x 4 KiB takes 74 us for its three passes over
// 128 MiB (312 and a copy of 40 before it when each warp read 32 rows' words 4 KiB
// apart and took 64 ballots a word); the columns of the slots that 256 writes
// touched 8.4 (126 then and 21 now by whole rows).
template <bool COPY>
__global__ void __launch_bounds__(256) tcopy_kernel(const uint4* __restrict__ src, uint64_t n, uint32_t Wd,
                                                    uint4* __restrict__ table, uint64_t* __restrict__ Tt,
                                                    uint64_t nblocks, const __grid_constant__ TcopyBlocks bl) {
  __shared__ uint32_t tile[64][33];
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t Ws = bl.count ? bl.slot_words : Wd;  // words of an entry: a slot, or the row
  const uint32_t chunks = (Ws + 31) / 32, U = Wd / 4;
  const uint64_t items = (bl.count ? bl.count : nblocks) * chunks;
  const uint64_t row_bits = static_cast<uint64_t>(Wd) * 32;
  const WarpTranspose transpose;
  for (uint64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const uint64_t kb = bl.count ? bl.kb[it / chunks] : it / chunks;
    const uint32_t wb = bl.count ? bl.slot[it / chunks] * Ws : 0u;  // first word, and past the last
    const uint32_t w0 = wb + static_cast<uint32_t>(it % chunks) * 32, we = wb + Ws;
    // thread: 16 bytes of rows threadIdx / 8 and 32 + threadIdx / 8
    const uint32_t r = threadIdx.x >> 3, u = threadIdx.x & 7u, uc = w0 / 4 + u;
    uint4 v[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
#pragma unroll
    for (uint32_t h = 0; h < 2; ++h) {
      const uint64_t row = 64 * kb + 32 * h + r;
      if (row < n && 4 * uc < we) v[h] = src[row * U + uc];
    }
    __syncthreads();  // the tile's last readers are done
#pragma unroll
    for (uint32_t h = 0; h < 2; ++h) {
      uint32_t* t = &tile[32 * h + r][4 * u];
      t[0] = v[h].x;
      t[1] = v[h].y;
      t[2] = v[h].z;
      t[3] = v[h].w;
      const uint64_t row = 64 * kb + 32 * h + r;
      if (COPY && row < n && uc < U) table[row * U + uc] = v[h];
    }
    __syncthreads();
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
      const uint32_t c = 4 * warp + i;
      if (w0 + c >= we) break;  // uniform over the warp
      const uint32_t lo = transpose(tile[lane][c]), hi = transpose(tile[32 + lane][c]);
      Tt[kb * row_bits + static_cast<uint64_t>(w0 + c) * 32 + lane] =
          static_cast<uint64_t>(lo) | (static_cast<uint64_t>(hi) << 32);
    }
  }
}

// src: the table itself, or (all blocks) device memory to copy to it as well
cudaError_t launch_tcopy(const tpir_db* db, const void* src, const TcopyBlocks& bl, cudaStream_t st) {
  const uint64_t nblocks = (db->n + 63) / 64;
  const uint64_t items = bl.count ? static_cast<uint64_t>(bl.count) * ((bl.slot_words + 31) / 32)
                                  : nblocks * ((db->Wd + 31) / 32);
  if (items == 0) return cudaSuccess;
  const uint32_t grid = static_cast<uint32_t>(
      std::min<uint64_t>(items, static_cast<uint64_t>(device_sm_count()) * 8));
  const uint4* s4 = static_cast<const uint4*>(src);
  uint4* t4 = reinterpret_cast<uint4*>(db->d_table);
  if (src == db->d_table)
    tcopy_kernel<false><<<grid, 256, 0, st>>>(s4, db->n, db->Wd, t4, db->d_tt, nblocks, bl);
  else
    tcopy_kernel<true><<<grid, 256, 0, st>>>(s4, db->n, db->Wd, t4, db->d_tt, nblocks, bl);
  count_launches();
  return cudaGetLastError();
}

}  // namespace

// Slots (of 64 buckets) up to which writes update a copy that only smaller batches use.
constexpr size_t kTcopyFewSlots = 16;

uint64_t tcopy_bytes(uint64_t n, uint32_t row_bytes) { return (n + 63) / 64 * 64 * row_bytes; }

cudaError_t tcopy_ensure(tpir_db* db, cudaStream_t st) {
  if (db->tt_valid) return cudaSuccess;
  if (!db->d_tt) {
    const uint64_t bytes = tcopy_bytes(db->n, db->row_bytes);
    const RelaxedCapture relaxed;  // (a read on another stream than the captured one)
    if (!db->tt_wanted) {  // only for the smaller batches: not if it would make memory scarce
      size_t free_b = 0, total_b = 0;
      if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || bytes > free_b / 4) {
        cudaGetLastError();
        db->tt_scarce = true;
        return cudaErrorMemoryAllocation;
      }
    }
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&db->d_tt), bytes);
    if (e != cudaSuccess) {
      db->d_tt = nullptr;
      if (e == cudaErrorMemoryAllocation) db->tt_skip = kTcopySkip;
      cudaGetLastError();
      return e;
    }
    db->tt_skip = 0;
    db->tt_scarce = false;
  }
  TcopyBlocks all{};
  cudaError_t e = launch_tcopy(db, db->d_table, all, st);
  // reads on other streams come after the copy as they come after a write
  if (e == cudaSuccess) e = note_write(db, st);
  if (e == cudaSuccess) db->tt_valid = true;
  if (e == cudaSuccess) order_after_writes(db, st);  // the read that comes next as well
  return e;
}

bool tcopy_load(tpir_db* db, const void* src, cudaStream_t st, cudaError_t* e) {
  // only where the copy is rebuilt anyway, from memory of this device that the
  // kernel can read by 16 bytes
  if (!db->d_tt || !db->tt_wanted || (reinterpret_cast<uintptr_t>(src) & 15)) return false;
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, src) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int dev = -1;
  if (at.type != cudaMemoryTypeDevice || cudaGetDevice(&dev) != cudaSuccess || dev != at.device) return false;
  const uint8_t* s8 = static_cast<const uint8_t*>(src);
  const uint64_t bytes = db->n * db->row_bytes;
  if (s8 < db->d_table + bytes && db->d_table < s8 + bytes) return false;  // overlapping: a plain copy
  TcopyBlocks all{};
  db->tt_skip = 0;
  db->tt_scarce = false;
  db->tt_valid = false;
  *e = launch_tcopy(db, src, all, st);
  if (*e == cudaSuccess) db->tt_valid = true;
  return true;
}

cudaError_t tcopy_after_load(tpir_db* db, cudaStream_t st) {
  db->tt_skip = 0;
  db->tt_scarce = false;
  if (!db->tt_wanted) db->rule.changed(copy_build_us(tcopy_bytes(db->n, db->row_bytes)));
  db->tt_valid = false;
  // (built on first use; where only smaller batches used it, again when it is worth it)
  return db->d_tt && db->tt_wanted ? tcopy_ensure(db, st) : cudaSuccess;
}

cudaError_t tcopy_after_moves(tpir_db* db, const MoveOp* ops, size_t nops, cudaStream_t st) {
  if (nops == 0) return cudaSuccess;
  const double build = copy_build_us(tcopy_bytes(db->n, db->row_bytes));
  if (!db->tt_valid) {
    if (nops > kTcopyFewSlots)
      db->rule.changed(build);
    else
      db->rule.wrote(kCopyUpdateUs, build);
    return cudaSuccess;
  }
  TcopyBlocks bl{};
  std::vector<uint64_t> kbs;
  kbs.reserve(nops);
  for (size_t i = 0; i < nops; ++i)
    if (ops[i].dst != kTmpSlot)  // (block, slot of the bucket)
      kbs.push_back(ops[i].dst / db->d / 64 * db->d + ops[i].dst % db->d);
  std::sort(kbs.begin(), kbs.end());
  kbs.erase(std::unique(kbs.begin(), kbs.end()), kbs.end());
  if (!db->tt_wanted && (kbs.size() > kTcopyFewSlots || db->rule.wrote(kCopyUpdateUs, build))) {
    db->rule.changed(build);  // as after a load
    db->tt_valid = false;
    return cudaSuccess;
  }
  uint32_t d = db->d;
  bl.slot_words = db->z / 4;
  if (kbs.size() > kTcopyMaxBlocks) {  // too many slots to list: their blocks, by whole rows
    for (uint64_t& k : kbs) k /= d;
    kbs.erase(std::unique(kbs.begin(), kbs.end()), kbs.end());
    d = 1;
    bl.slot_words = db->Wd;
  }
  if (kbs.size() > kTcopyMaxBlocks) return launch_tcopy(db, db->d_table, bl, st);  // rebuild it all
  bl.count = static_cast<uint32_t>(kbs.size());
  for (size_t i = 0; i < kbs.size(); ++i) {
    bl.kb[i] = kbs[i] / d;
    bl.slot[i] = static_cast<uint8_t>(kbs[i] % d);
  }
  return launch_tcopy(db, db->d_table, bl, st);
}

}  // namespace tpir
