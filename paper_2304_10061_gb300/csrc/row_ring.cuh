// Per-warp shared-memory rings over the edges of a row, filled by cp.async (row kernels).
#pragma once

#include <cuda_runtime.h>

namespace alg {

// ---------------------------------------------------------------------------
// Asynchronous copies of an edge's rows into shared memory, so that a warp has
// several edges' loads in flight without holding them in registers (the row
// kernels keep 64 to 100 floats of per-channel state, which leaves 8 to 16
// warps per SM: with one or two edges in flight each they waited on latency).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// `bytes` (even) contiguous bytes at src to dst (16-byte aligned) by the warp; `al` = the low four bits of src and
// bytes or'ed: 16-byte copies when they are zero, else 4-byte ones, else plain 2-byte copies (latent
// widths that are odd in bf16)
__device__ __forceinline__ void warp_copy(unsigned char* dst, const unsigned char* src, int bytes, unsigned al) {
  const int lane = threadIdx.x & 31;
  if (al == 0) {
    for (int k = lane * 16; k < bytes; k += 512) cp_async16(dst + k, src + k);
  } else if ((al & 3) == 0) {
    for (int k = lane * 4; k < bytes; k += 128) cp_async4(dst + k, src + k);
  } else {
    for (int k = lane * 2; k < bytes; k += 64)
      *reinterpret_cast<unsigned short*>(dst + k) = *reinterpret_cast<const unsigned short*>(src + k);
  }
}

__host__ __device__ constexpr int round16(int x) { return (x + 15) / 16 * 16; }

// A warp's ring over its row's edges: D stages of STAGE bytes.  copy(e, slot) queues edge e's rows into
// a slot; for each edge in order, use(e, slot) runs once the edge's rows have arrived, with the next
// D - 1 edges queued.  ring_begin queues the first edges (no lane may still read the ring), ring_loop
// does the rest, so work that needs none of the rows can go between.
template <int D, int STAGE, typename Copy>
__device__ __forceinline__ void ring_begin(unsigned char* ring, int rb, int re, Copy&& copy) {
#pragma unroll
  for (int p = 0; p < D - 1; ++p) {
    if (rb + p < re) copy(rb + p, ring + p * STAGE);
    cp_async_commit();
  }
}
template <int D, int STAGE, typename Copy, typename Use>
__device__ __forceinline__ void ring_loop(unsigned char* ring, int rb, int re, Copy&& copy, Use&& use) {
  int slot = 0;
  for (int e = rb; e < re; ++e) {
    cp_async_wait<D - 2>();
    __syncwarp();   // every lane's copies of edge e have landed, and no lane still reads the slot before it
    const int nslot = (slot + D - 1) % D;
    if (e + D - 1 < re) copy(e + D - 1, ring + nslot * STAGE);
    cp_async_commit();
    use(e, ring + slot * STAGE);
    slot = (slot + 1) % D;
  }
}
template <int D, int STAGE, typename Copy, typename Use>
__device__ __forceinline__ void ring_over(unsigned char* ring, int rb, int re, Copy&& copy, Use&& use) {
  ring_begin<D, STAGE>(ring, rb, re, copy);
  ring_loop<D, STAGE>(ring, rb, re, copy, use);
}

}  // namespace alg
