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

// ---- EPI_HEAD_WIDE: the adjoint head of x = u silu(z) in a GEMM's epilogue ----
// Two warps share a quarter's rows, warp h the 32-column chunks h, h + 2, ...; a thread has one row.
// The row sum is that of head_bwd_kernel: 32 partial sums, partial l over the columns 4 l .. 4 l + 3 of
// every 128 in ascending order, then halving sums over l.  Chunk c holds the partials 8 (c mod 4) ..
// + 7, so warp h owns the partials 8 h .. 8 h + 7 (d0) and 16 + 8 h .. (d1), and the first halving
// stays in a thread; the second takes warp 1's eight values through its staging box.  A CTA runs the
// column tiles of a row block one after another.
// Bound: as the GEMM's other epilogues.  Without it the GEMM writes xbar in float32 and head_bwd_kernel
// reads it and z and writes zbar at 90 % of HBM: ms per step, separate / fused, 3-layer model, 65,536
// atoms bf16 36.5 / 34.1, 16,384 atoms fp8 10.21 / 9.67; 1024-wide MLPs, 16,411 atoms bf16 6.17 / 5.90;
// 256-wide, 3,072 atoms TF32 1.162 / 1.110.
struct HeadSums {
  float d0[8], d1[8];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 8; ++k) d0[k] = d1[k] = 0.0f;
  }
};
// one element: adds xbar silu(z) to its partial and returns zbar
__device__ __forceinline__ float head_elem(float xb, float z, float ue, float& d) {
  const float s = epi_sigmoid(z);
  d = fmaf(xb * z, s, d);
  return xb * ue * s * (1.0f + z * (1.0f - s));
}
// After a row block's last column tile: `xbox` warp 1's staging box (1 KB of it), `ready` / `used`
// barriers of one arrival, `nrow` the row blocks this CTA finished before; ubar null: no row.
// False: a wait ran out.
__device__ __forceinline__ bool head_finish(int h, int lane, const HeadSums& hs, uint8_t* xbox, uint64_t* ready,
                                            uint64_t* used, int nrow, float* ubar) {
  float a[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) a[k] = hs.d0[k] + hs.d1[k];
  float* x = reinterpret_cast<float*>(xbox) + lane;
  if (h != 0) {
    if (lane == 0) bulk_wait_read0();   // the box's last store has been read
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; ++k) x[32 * k] = a[k];
    __syncwarp();
    if (lane == 0) mbar_arrive(ready);
    return true;
  }
  if (!mbar_wait(ready, nrow & 1)) return false;
#pragma unroll
  for (int k = 0; k < 8; ++k) a[k] += x[32 * k];
  __syncwarp();
  if (lane == 0) mbar_arrive(used);
#pragma unroll
  for (int w = 4; w > 0; w >>= 1)
#pragma unroll
    for (int k = 0; k < w; ++k) a[k] += a[k + w];
  if (ubar) *ubar += a[0];
  return true;
}
// before warp 1's first store of a row block: warp 0 has read the partials of the one before
__device__ __forceinline__ bool head_start(int h, uint64_t* used, int nrow) {
  return h == 0 || nrow == 0 || mbar_wait(used, (nrow - 1) & 1);
}

}  // namespace alg
