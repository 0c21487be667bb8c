// Warp-level TF32 products (m16n8k8) with a hi / lo split of FP32 operands, and
// the block layout of their tables: shared by the x-update kernels
// (contract_admm.cu, contract_warp.cu).  Internal header: not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

// TF32 split: hi = x rounded to the TF32 grid (to nearest, ties away from zero: the
// same value as cvt.rna), lo = x - hi exactly, passed to the MMA as raw FP32 bits, of
// which the tensor core reads the TF32 part (|lo| <= 2^-11 |x|, so what is dropped is
// below 2^-21 |x|).
__device__ __forceinline__ void split_fast(float x, unsigned& hi, unsigned& lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Copies of src [nclass][rows][ld] (cols columns) in 8 x 8 blocks [rb][cb][64] (zero
// padding), the words of a block permuted as
//   word(i, j) = 32 (j / 4) + 4 ((i + 4 (j / 4)) mod 8) + j mod 4,
// so that fragments of the block and of its transpose load without bank conflicts.
static __global__ void k_block_rows(const float* __restrict__ src, int rows, int cols, int ld, int rb, int cb,
                                    float* __restrict__ dst, int nclass) {
  const size_t per = (size_t)rb * cb * 64, total = per * nclass;
  for (size_t d = (size_t)blockIdx.x * blockDim.x + threadIdx.x; d < total; d += (size_t)gridDim.x * blockDim.x) {
    const size_t c = d / per;
    const int rem = (int)(d - c * per), blk = rem >> 6, w = rem & 63;
    const int br = blk / cb, bc = blk - br * cb;
    const int half = w >> 5, q = w & 31;
    const int r = 8 * br + (((q >> 2) - 4 * half) & 7), col = 8 * bc + 4 * half + (q & 3);
    dst[d] = (r < rows && col < cols) ? src[c * (size_t)rows * ld + (size_t)r * ld + col] : 0.f;
  }
}
