// The order of importances: fp32 bit patterns as order-preserving unsigned keys.
#pragma once

#include <stdint.h>

namespace sg {

// Takes the raw bit pattern: the row is read as uint32 so that no float instruction (and no
// flush-to-zero of subnormals) ever touches the values.
__device__ __forceinline__ uint32_t order_key(uint32_t u) {
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ uint32_t key_to_bits(uint32_t k) { return (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k; }
constexpr uint32_t kKeyNegInf = 0x007fffffu, kKeyPosInf = 0xff800000u;

}  // namespace sg
