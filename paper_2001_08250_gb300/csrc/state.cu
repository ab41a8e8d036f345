// Server-state kernels for sm_103a.
//
//  apply_moves_param_kernel, settled_moves_kernel  the device half of a cuckoo
//                      write (Section 5.3): the host computes where every
//                      touched item ends up and emits an ordered list of slot
//                      copies (with a one-slot temporary to break cycles),
//                      payload writes and slot clears (FIFO collection).  A
//                      list that fits the kernel parameters is run in order by
//                      one CTA; a longer one is settled first (cuckoo.cpp:
//                      what each slot holds in the end) and its slots are
//                      written by a CTA each.
//  bloom_*_kernel      Section 7: OR a write's interest vector (k positions or
//                      a whole vector) into the current delta, and form the
//                      global interest vector as the OR of the window's deltas.
#include <algorithm>

#include "tpir_internal.h"

namespace tpir {
namespace {

constexpr uint32_t kMoveThreads = 256;

// Slot writes that do not depend on one another (settle_moves), one column of
// the grid each: from a message, a table slot that no write of the list touches,
// or the saved slots (and the saving itself: kinds 3 and 4), or zeros.
// Bound by latency: 256 writes of 1 KiB take 3.6 us (188 in order in one CTA,
// 0.7 us a write).  A large slot is spread over CTAs: one write of 1 MiB or 16 MiB,
// the call with its copies to the device, takes 72 and 400 us (150 and 2 250 with 64
// threads a slot, 111 and 1 270 in order with 256).
__global__ void __launch_bounds__(kMoveThreads) settled_moves_kernel(uint8_t* __restrict__ table, uint32_t z,
                                                                     const MoveOp* __restrict__ ops,
                                                                     const uint8_t* __restrict__ payloads,
                                                                     uint8_t* __restrict__ saved) {
  const MoveOp op = ops[blockIdx.x];
  uint4* dst = reinterpret_cast<uint4*>(op.kind == 4 ? saved + op.dst * z : table + op.dst * z);
  const uint8_t* s8 = op.kind == 1 ? payloads + op.src * z : op.kind == 3 ? saved + op.src * z : table + op.src * z;
  const uint4* src = reinterpret_cast<const uint4*>(s8);
  const uint32_t z4 = z / 16, j0 = blockIdx.y * blockDim.x + threadIdx.x, step = gridDim.y * blockDim.x;
  if (op.kind == 2)
    for (uint32_t j = j0; j < z4; j += step) dst[j] = make_uint4(0u, 0u, 0u, 0u);
  else
    for (uint32_t j = j0; j < z4; j += step) dst[j] = src[j];
}

// The ordered moves of a small batch of writes, with the move list and the new
// messages passed by value in the kernel parameters: no staging buffer, no
// copy before the launch, so a single write costs one launch.
template <typename PM>
__global__ void __launch_bounds__(256) apply_moves_param_kernel(uint8_t* __restrict__ table,
                                                                uint32_t z,
                                                                const __grid_constant__ PM m,
                                                                uint8_t* __restrict__ tmp) {
  const uint32_t z4 = z / 16;
  for (uint32_t i = 0; i < m.nops; ++i) {
    const MoveOp op = m.ops[i];
    uint4* dst = reinterpret_cast<uint4*>(op.dst == kTmpSlot ? tmp : table + op.dst * z);
    if (op.kind == 2) {
      for (uint32_t j = threadIdx.x; j < z4; j += blockDim.x) dst[j] = make_uint4(0u, 0u, 0u, 0u);
    } else if (op.kind == 1) {
      const uint4* src = reinterpret_cast<const uint4*>(m.payload + op.src * z);
      for (uint32_t j = threadIdx.x; j < z4; j += blockDim.x) dst[j] = src[j];
    } else {
      const uint4* src = reinterpret_cast<const uint4*>(op.src == kTmpSlot ? tmp : table + op.src * z);
      for (uint32_t j = threadIdx.x; j < z4; j += blockDim.x) dst[j] = src[j];
    }
    __syncthreads();  // the next op may read what this one wrote
  }
}

__global__ void bloom_set_kernel(uint64_t* __restrict__ delta, const uint64_t* __restrict__ pos,
                                 uint64_t count) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t p = pos[i];
    atomicOr(reinterpret_cast<unsigned long long*>(delta + (p >> 6)), 1ull << (p & 63));
  }
}

__global__ void bloom_or_kernel(uint64_t* __restrict__ delta, const uint64_t* __restrict__ vec,
                                uint64_t m) {
  const uint64_t words = (m + 63) / 64;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < words;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t v = vec[i];
    if (i == words - 1 && (m & 63)) v &= (1ull << (m & 63)) - 1;
    delta[i] |= v;
  }
}

__global__ void bloom_union_kernel(const uint64_t* __restrict__ deltas, uint32_t window,
                                   uint64_t words, uint64_t* __restrict__ out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < words;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t v = 0;
    for (uint32_t j = 0; j < window; ++j) v |= deltas[j * words + i];
    out[i] = v;
  }
}

}  // namespace

cudaError_t launch_settled_moves(uint8_t* table, uint32_t z, const MoveOp* ops, uint32_t nsave,
                                 uint32_t nops, const uint8_t* payloads, uint8_t* saved,
                                 cudaStream_t st) {
  // a thread per 16 bytes of a slot, in up to 1 024 CTAs
  const uint32_t z4 = z / 16, threads = std::min(kMoveThreads, (z4 + 31) / 32 * 32);
  const uint32_t y = std::min(1024u, (z4 + threads - 1) / threads);
  if (nsave) {
    settled_moves_kernel<<<dim3(nsave, y), threads, 0, st>>>(table, z, ops, payloads, saved);
    count_launches();
  }
  if (nops > nsave) {
    settled_moves_kernel<<<dim3(nops - nsave, y), threads, 0, st>>>(table, z, ops + nsave, payloads, saved);
    count_launches();
  }
  return cudaGetLastError();
}

cudaError_t launch_apply_moves_param(uint8_t* table, uint32_t z, const ParamMoves& m, uint8_t* tmp,
                                     cudaStream_t st) {
  if (m.nops == 0) return cudaSuccess;
  apply_moves_param_kernel<ParamMoves><<<1, 256, 0, st>>>(table, z, m, tmp);
  count_launches();
  return cudaGetLastError();
}

cudaError_t launch_apply_moves_param(uint8_t* table, uint32_t z, const ParamMovesS& m, uint8_t* tmp,
                                     cudaStream_t st) {
  if (m.nops == 0) return cudaSuccess;
  apply_moves_param_kernel<ParamMovesS><<<1, 256, 0, st>>>(table, z, m, tmp);
  count_launches();
  return cudaGetLastError();
}

cudaError_t launch_bloom_set(uint64_t* delta, const uint64_t* pos, uint64_t count,
                             cudaStream_t st) {
  if (count == 0) return cudaSuccess;
  const uint64_t blocks = (count + 255) / 256;
  bloom_set_kernel<<<static_cast<uint32_t>(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(delta, pos,
                                                                                        count);
  count_launches();
  return cudaGetLastError();
}

cudaError_t launch_bloom_or(uint64_t* delta, const uint64_t* vec, uint64_t m, cudaStream_t st) {
  const uint64_t words = (m + 63) / 64;
  const uint64_t blocks = (words + 255) / 256;
  bloom_or_kernel<<<static_cast<uint32_t>(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(delta, vec,
                                                                                       m);
  count_launches();
  return cudaGetLastError();
}

cudaError_t launch_bloom_union(const uint64_t* deltas, uint32_t window, uint64_t words,
                               uint64_t* out, cudaStream_t st) {
  const uint64_t blocks = (words + 255) / 256;
  bloom_union_kernel<<<static_cast<uint32_t>(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(
      deltas, window, words, out);
  count_launches();
  return cudaGetLastError();
}

}  // namespace tpir
