// Epilogue staging of the tcgen05 GEMMs: 32 x 32 boxes (a warp's 32 accumulator rows x 32 columns)
// in swizzled shared memory, moved by TMA, so that global memory sees whole rows of a box instead of
// one 16-byte piece per lane and instruction (a row per lane touches 32 lines with every access).
#pragma once

#include <cuda.h>

#include <cstdint>

#include "epilogue.cuh"
#include "tc_ptx.cuh"

namespace alg {

// --- epilogue staging: 32 x 32 boxes moved by TMA --------------------------
// bf16 box rows are 64 bytes (64-byte swizzle), float32 box rows 128 bytes
// (128-byte swizzle); the 16-byte unit u of row r sits at unit u ^ f(r) so the
// row-per-lane accesses spread over all banks.
__device__ __forceinline__ uint32_t sw64(int r, int u) { return r * 64 + ((u ^ ((r >> 1) & 3)) << 4); }
__device__ __forceinline__ uint32_t sw128(int r, int u) { return r * 128 + ((u ^ (r & 7)) << 4); }

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* tm, const void* src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(tm)),
               "r"(smem_u32(src)), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void st_bf16_row(uint8_t* box, int r, const float (&v)[32]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    uint4 x = make_uint4(pack_bf16x2(v[8 * u + 0], v[8 * u + 1]), pack_bf16x2(v[8 * u + 2], v[8 * u + 3]),
                         pack_bf16x2(v[8 * u + 4], v[8 * u + 5]), pack_bf16x2(v[8 * u + 6], v[8 * u + 7]));
    *reinterpret_cast<uint4*>(box + sw64(r, u)) = x;
  }
}
__device__ __forceinline__ void ld_bf16_row(const uint8_t* box, int r, float (&v)[32]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    uint4 x = *reinterpret_cast<const uint4*>(box + sw64(r, u));
    uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      float2 f = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w[t]));
      v[8 * u + 2 * t] = f.x;
      v[8 * u + 2 * t + 1] = f.y;
    }
  }
}
__device__ __forceinline__ void st_f32_row(uint8_t* box, int r, const float (&v)[32]) {
#pragma unroll
  for (int u = 0; u < 8; ++u)
    *reinterpret_cast<float4*>(box + sw128(r, u)) = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
}
__device__ __forceinline__ void ld_f32_row(const uint8_t* box, int r, float (&v)[32]) {
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    float4 x = *reinterpret_cast<const float4*>(box + sw128(r, u));
    v[4 * u] = x.x; v[4 * u + 1] = x.y; v[4 * u + 2] = x.z; v[4 * u + 3] = x.w;
  }
}

// 16 columns (half hh of a 32-column box row) into the swizzled staging boxes.
__device__ __forceinline__ void st_bf16_half(uint8_t* box, int r, int hh, const float (&v)[16]) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    uint4 x = make_uint4(pack_bf16x2(v[8 * u + 0], v[8 * u + 1]), pack_bf16x2(v[8 * u + 2], v[8 * u + 3]),
                         pack_bf16x2(v[8 * u + 4], v[8 * u + 5]), pack_bf16x2(v[8 * u + 6], v[8 * u + 7]));
    *reinterpret_cast<uint4*>(box + sw64(r, 2 * hh + u)) = x;
  }
}
__device__ __forceinline__ void st_f32_half(uint8_t* box, int r, int hh, const float (&v)[16]) {
#pragma unroll
  for (int u = 0; u < 4; ++u)
    *reinterpret_cast<float4*>(box + sw128(r, 4 * hh + u)) = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
}

struct EpiMaps {
  CUtensorMap out, pre, add;
};

// Raw bf16 words of one 32-column row of a swizzled bf16 32x32 box (16 words).
__device__ __forceinline__ void ld_bf16_row_raw(const uint8_t* box, int r, uint32_t (&w)[16]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const uint4 x = *reinterpret_cast<const uint4*>(box + sw64(r, u));
    w[4 * u] = x.x; w[4 * u + 1] = x.y; w[4 * u + 2] = x.z; w[4 * u + 3] = x.w;
  }
}
// element j (0..31) of such a row
__device__ __forceinline__ float bf16_word_elem(const uint32_t (&w)[16], int j) {
  const uint32_t x = w[j >> 1];
  return __uint_as_float((j & 1) ? (x & 0xffff0000u) : (x << 16));
}

}  // namespace alg
