// hy_tc.cuh -- what the tensor-core kernels share: operands in shared memory
// (K-major, no swizzle: core matrices of 8 rows x 16 bytes, consecutive cores
// along K 128 bytes apart, along M/N `sbo` bytes apart) and the split of an FP32
// value into two TF32 ones.
#pragma once

#include <cstdint>

namespace hy {
namespace k {

__device__ __forceinline__ uint32_t saddr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// byte offset of element (row, k) in a K-major no-swizzle operand
__device__ __forceinline__ uint32_t kmaj(int row, int k, uint32_t sbo)
{
    return uint32_t(row >> 3) * sbo + uint32_t(k >> 2) * 128u + uint32_t(row & 7) * 16u +
           uint32_t(k & 3) * 4u;
}

__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t sbo)
{
    return uint64_t((addr >> 4) & 0x3FFFu) | (uint64_t(128u >> 4) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (uint64_t(1) << 46);
}

__device__ __forceinline__ void split(float x, float &hi, float &lo)
{
    hi = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
    lo = x - hi;
}

// the same with hi rounded to nearest: lo may have either sign, so that what the
// tensor cores cut off it does not add up
__device__ __forceinline__ void split_rn(float x, float &hi, float &lo)
{
    hi = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
    lo = x - hi;
}

// one lane of a converged warp, the same one each time
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}

}  // namespace k
}  // namespace hy
