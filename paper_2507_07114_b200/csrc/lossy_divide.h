// Division by a number that the host knows. (No CUDA header: tests/test_divide.py compiles it for the host.)
#pragma once
#include <stdint.h>

namespace lossy {

// x / d for a d that the host knows: the high half of x times 2^64 / d rounded up, exact for every 32-bit x and d (the product is too
// large by less than x d < 2^64). Two multiply-adds for a division's twenty and more instructions.
__host__ inline uint64_t magic_of(uint32_t d) { return d > 1u ? ~0ull / d + 1ull : 0ull; }
__host__ __device__ __forceinline__ uint32_t divide_by(uint32_t x, uint32_t d, uint64_t magic) {
  const uint64_t low = (uint64_t)x * (uint32_t)magic;
  return d > 1u ? (uint32_t)(((uint64_t)x * (uint32_t)(magic >> 32) + (low >> 32)) >> 32) : x;
}

}  // namespace lossy
