// Warp-level tensor-core products in TF32 with FP32 accumulation, and the
// head/tail split of their operands: x = head + tail with both TF32, a*b summed
// as tail_a*head_b + head_a*tail_b + head_a*head_b.  A tail is at most 2^-11 of
// its operand and keeps it to one unit of FP32 (2^-23): the dropped tail*tail
// term is at most 2^-22 of a product, the operands' last units another 2^-22.
#pragma once

#include <cstdint>
#include <cstring>

namespace ams {

__host__ __device__ __forceinline__ uint32_t f32_bits(float x) {
    uint32_t u;
    memcpy(&u, &x, sizeof u);
    return u;
}
__host__ __device__ __forceinline__ float f32_of_bits(uint32_t u) {
    float x;
    memcpy(&x, &u, sizeof x);
    return x;
}
// The head is the nearest TF32 value (ties away).  What is left is exact in FP32
// with at most 12 significant bits; the tail is its 11 leading ones, cut off
// here: what an MMA makes of an operand with more bits is not specified.  Four
// operations at the ALU's rate; two cvt.rna instructions, at a quarter of it,
// made the kernels that split on the fly issue-bound (coarse products at 32
// right-hand sides, N_c = 24,576: 322 -> 272 us).  A NaN or infinity has a NaN tail.
__host__ __device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
    hi = (f32_bits(x) + 0x1000u) & 0xffffe000u;
    lo = f32_bits(x - f32_of_bits(hi)) & 0xffffe000u;
}
// d += a b, a 16x8 (row), b 8x8 (col), TF32 in, FP32 accumulate
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

}  // namespace ams
