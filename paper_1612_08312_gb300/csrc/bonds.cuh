// bonds.cuh -- decisions of bonds from their random bytes, shared by the
// pyrochlore and the generic-lattice sweeps: four bytes of a word compared at
// a time (Ising), and the fast exponential of the n-vector shortcut.
#pragma once

#include "pyro_internal.cuh"

namespace pyro {

// Bytewise unsigned a < b: bit 7 of each byte of the result.
__device__ __forceinline__ uint32_t bytes_lt(uint32_t a, uint32_t b)
{
    const uint32_t d = (a | 0x80808080u) - (b & 0x7F7F7F7Fu);  // bit 7: low 7 bits of a >= those of b
    return ((~(a ^ b) & ~d) | (~a & b)) & 0x80808080u;
}

// Bytewise a == b: bit 7 of each byte.
__device__ __forceinline__ uint32_t bytes_eq(uint32_t a, uint32_t b)
{
    const uint32_t t = a ^ b;
    return ~(((t & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | t) & 0x80808080u;
}

// Bit 7 of the four bytes -> four low bits.
__device__ __forceinline__ uint32_t byte_flags_to_nibble(uint32_t f) { return (((f >> 7) * 0x204081u) >> 21) & 0xFu; }

// Threshold of a bond: active iff its 32-bit uniform w < thr (thr <= 2^32).
// w's top byte comes from the BOND stream, its low 24 bits (only needed on
// a tie of the top bytes) from the TIE stream.
struct ByteCompare {
    uint32_t t8, t24;
    bool all, none;
    __device__ __forceinline__ explicit ByteCompare(uint64_t thr)
        : t8((uint32_t)(thr >> 24)), t24((uint32_t)(thr & 0xFFFFFFu)), all(thr >= (1ull << 32)), none(thr == 0) {}
};

// 2^x, relative error at most 2^-22 (PTX ISA, ex2.approx.ftz.f32).
__device__ __forceinline__ float exp2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Margin of the n-vector bond shortcut, in units of 1/256 of probability, for
// a product of projections given to a few 2^-24 relative (see vector.cu).
constexpr float SHORTCUT_MARGIN = 1e-3f;

}  // namespace pyro
