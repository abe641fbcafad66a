// Layout of the split-bf16 operand of the tensor-core transforms, shared by the kernels that write it:
// [parity][m tile of 128 rows][K tile of 64][hi | lo][128 x 64 bf16, K-major 128-byte swizzle].
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace lag {

constexpr int TM = 128;              // rows per tile (MMA M)
constexpr int TK = 64;               // K per tile (one 128-byte swizzle atom of bf16)
constexpr int A_TILE = TM * TK * 2;  // 16 KB

// element (r, k) of a rows x 64 tile in the K-major SWIZZLE_128B layout (byte offset)
__host__ __device__ __forceinline__ uint32_t swz(int r, int k) {
  return (uint32_t)r * 128u + ((uint32_t)((k >> 3) ^ (r & 7)) << 4) + (uint32_t)(k & 7) * 2u;
}

__device__ __forceinline__ uint16_t bf16_bits(float f) {
  __nv_bfloat16 b = __float2bfloat16_rn(f);
  return *reinterpret_cast<uint16_t *>(&b);
}

// split f into bf16 hi + bf16 lo in float32 arithmetic (FP64 throughput is 1/61 of FP32 on this part;
// hi + lo keeps 16 significant bits)
__device__ __forceinline__ void split2f(float f, uint16_t &hi, uint16_t &lo) {
  __nv_bfloat16 h = __float2bfloat16_rn(f);
  hi = *reinterpret_cast<uint16_t *>(&h);
  lo = bf16_bits(f - __bfloat162float(h));
}

// an operand area (null: none) and its extent
struct TcOperand {
  uint8_t *a = nullptr;
  int ku = 0;   // columns of parity 0 in a parity-permuted row
  int nks = 0;  // K tiles
  int nmt = 0;  // m tiles
};

}  // namespace lag
