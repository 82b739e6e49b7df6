// Device helpers shared by the kernel files: the edge and relaxation keys, the block-wide scan and the weight counters.
#pragma once
#include "internal.h"

namespace mstgpu {

__device__ __forceinline__ u64 edge_key(uint32_t w, uint32_t id) { return ((u64)w << 32) | (u64)id; }

// Relaxation key of an edge as seen from one end (see KeyLayout).
__device__ __forceinline__ u64 relax_key(const KeyLayout &kl, uint32_t w, uint32_t id, uint32_t other) {
  return kl.packed ? (((u64)w << (kl.idbits + kl.vbits)) | ((u64)id << kl.vbits) | (u64)other) : edge_key(w, id);
}
__device__ __forceinline__ uint32_t key_edge_id(const KeyLayout &kl, u64 key) {
  return kl.packed ? (uint32_t)((key >> kl.vbits) & ((1ULL << kl.idbits) - 1)) : (uint32_t)key;
}
// The layout with `packed` decided on the device: where the largest weight
// *max_w leaves room for the id and the far end (max_w == nullptr: kl as is).
__device__ __forceinline__ KeyLayout resolve_layout(KeyLayout kl, const uint32_t *max_w) {
  if (max_w) {
    const uint32_t mw = __ldcg(max_w);
    kl.packed = (mw ? 32 - __clz(mw) : 0) + kl.idbits + kl.vbits <= 63;
  }
  return kl;
}
// Do two keys name the same edge (the 2-cycle test)?
__device__ __forceinline__ bool same_edge(const KeyLayout &kl, u64 a, u64 b) {
  return kl.packed ? (a >> kl.vbits) == (b >> kl.vbits) : a == b;
}

// Block solves: bits of a position among a graph's m edges (m > 0), and the
// weights from which on its keys take 64 bits.
__device__ __forceinline__ uint32_t block_pos_bits(uint32_t m) { return m > 1 ? 32 - __clz(m - 1) : 1; }
__device__ __forceinline__ uint32_t block_weight_limit(uint32_t m) { return (1u << (31 - block_pos_bits(m))) - 1u; }

__device__ __forceinline__ u64 mix64(u64 z) {  // splitmix64 finaliser
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

// Output #i of the splitmix64 sequence whose state starts at `state`
// (Steele, Lea, Flood, OOPSLA 2014).
__device__ __forceinline__ u64 splitmix64_at(u64 state, u64 i) {
  return mix64(state + (i + 1ULL) * 0x9e3779b97f4a7c15ULL);
}

// Exclusive block-wide scan of one uint32 per thread (B threads; s_warp holds
// B / 32 + 1 words).
template <int B = 256>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t &total, uint32_t *s_warp) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const uint32_t wv = lane < B / 32 ? s_warp[lane] : 0u;
    uint32_t wi = wv;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < B / 32) s_warp[lane] = wi - wv;
    if (lane == B / 32 - 1) s_warp[B / 32] = wi;
  }
  __syncthreads();
  total = s_warp[B / 32];
  return s_warp[wid] + incl - x;
}

// Copies the device state into the mapped host mirror, then publishes seq in the
// mapped flag word: by one block, behind its own stores and all it has seen.
// The system-scope fence orders them and the mirror's words before the flag.
__device__ __forceinline__ void publish_state(const Readback &rb) {
  static_assert(sizeof(DevState) % 4 == 0, "DevState is copied in words");
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < (uint32_t)(sizeof(DevState) / 4); i += blockDim.x)
    reinterpret_cast<volatile uint32_t *>(rb.mirror)[i] = __ldcg(reinterpret_cast<const uint32_t *>(rb.state) + i);
  __threadfence_system();
  __syncthreads();
  if (threadIdx.x == 0) *reinterpret_cast<volatile uint32_t *>(rb.flag) = rb.seq;
}

// Adds this thread's sum of chosen weights into a spread counter: one atomic
// per warp (all 32 lanes call together).
__device__ __forceinline__ void wsum_add(u64 *wsum, u64 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (wsum && (threadIdx.x & 31) == 0 && v)
    atomicAdd(reinterpret_cast<unsigned long long *>(wsum) +
                  ((blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) & (WSUM_SLOTS - 1)),
              (unsigned long long)v);
}

}  // namespace mstgpu
