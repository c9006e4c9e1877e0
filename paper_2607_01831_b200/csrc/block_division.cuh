// Division by the tokens of a block, without a division instruction.  Plain C++, so that it can be checked on the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define LYNX_BD_HD __host__ __device__ __forceinline__
#else
#define LYNX_BD_HD inline
#endif

namespace lynx {

// t / n = (t * mul >> 32) >> shift for 0 <= t < 2^31, 2 <= n < 2^31: with l = ceil(log2 n) and mul = floor(2^(31 + l) / n) + 1
// the error mul * n - 2^(31 + l) is in (0, 2^l], which 31 bits of t cannot carry to the next quotient.  (Granlund and Montgomery,
// Division by Invariant Integers using Multiplication, 1994.)
struct BlockDiv {
  uint32_t mul, shift;
};
inline BlockDiv block_div(int32_t n) {
  uint32_t l = 1;
  while ((1ll << l) < n) ++l;
  return {(uint32_t)((1ull << (31 + l)) / (uint32_t)n + 1), l - 1};
}
LYNX_BD_HD int32_t quotient(int32_t t, BlockDiv d) { return (int32_t)((uint32_t)(((uint64_t)(uint32_t)t * d.mul) >> 32) >> d.shift); }

}  // namespace lynx
