// Two float32 values in a 64-bit register: sm_100a adds, multiplies and fuses both in one instruction, each rounded as the
// scalar operation rounds it.  What it saves is issue slots, not cycles of the float32 pipe.
#ifndef DETAG_PACKED_CUH
#define DETAG_PACKED_CUH

#include <cstdint>

namespace detag {

struct F2 {
  unsigned long long bits;
};

__device__ __forceinline__ F2 pack2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.bits) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 both(float a) { return pack2(a, a); }
__device__ __forceinline__ void unpack2(F2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.bits)); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.bits) : "l"(a.bits), "l"(b.bits), "l"(c.bits));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.bits) : "l"(a.bits), "l"(b.bits));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.bits) : "l"(a.bits), "l"(b.bits));
  return r;
}
// a - b
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, both(-1.0f), a); }

}  // namespace detag
#endif  // DETAG_PACKED_CUH
