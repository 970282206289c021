// Carry chains over 32-bit words.  On the device each call is one instruction
// of a chain on the carry flag (a multiply-add takes its low and high call
// together); ptxas turns the flag into predicates, so that independent chains
// interleave.  A 64-bit sum per word takes about three times the
// instructions.  The host definitions, for CPU tests of the code built on
// them, keep the flag in a variable.
#pragma once

#include <stdint.h>

namespace ozlu {

#if defined(__CUDA_ARCH__)
#define OZ_CHAIN(name, ins)                                                           \
    __device__ __forceinline__ uint32_t name(uint32_t a, uint32_t b) {                \
        uint32_t r;                                                                   \
        asm volatile(ins " %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));                  \
        return r;                                                                     \
    }
#define OZ_CHAIN3(name, ins)                                                          \
    __device__ __forceinline__ uint32_t name(uint32_t a, uint32_t b, uint32_t c) {    \
        uint32_t r;                                                                   \
        asm volatile(ins " %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));      \
        return r;                                                                     \
    }
OZ_CHAIN(add_first, "add.cc.u32")    // a + b, sets the flag
OZ_CHAIN(add_next, "addc.cc.u32")    // a + b + flag, sets the flag
OZ_CHAIN(add_last, "addc.u32")       // a + b + flag
OZ_CHAIN3(mad_lo_first, "mad.lo.cc.u32")   // low word of a b, plus c, sets the flag
OZ_CHAIN3(mad_lo_next, "madc.lo.cc.u32")   // ... plus the flag
OZ_CHAIN3(mad_hi_next, "madc.hi.cc.u32")   // high word of a b, plus c and the flag
#undef OZ_CHAIN
#undef OZ_CHAIN3
#else
static thread_local uint32_t oz_carry_flag;
__device__ __forceinline__ uint32_t oz_chain(uint64_t s) {
    oz_carry_flag = (uint32_t)(s >> 32);
    return (uint32_t)s;
}
__device__ __forceinline__ uint32_t add_first(uint32_t a, uint32_t b) { return oz_chain((uint64_t)a + b); }
__device__ __forceinline__ uint32_t add_next(uint32_t a, uint32_t b) { return oz_chain((uint64_t)a + b + oz_carry_flag); }
__device__ __forceinline__ uint32_t add_last(uint32_t a, uint32_t b) { return a + b + oz_carry_flag; }
__device__ __forceinline__ uint32_t mad_lo_first(uint32_t a, uint32_t b, uint32_t c) {
    return oz_chain((uint64_t)(uint32_t)(a * b) + c);
}
__device__ __forceinline__ uint32_t mad_lo_next(uint32_t a, uint32_t b, uint32_t c) {
    return oz_chain((uint64_t)(uint32_t)(a * b) + c + oz_carry_flag);
}
__device__ __forceinline__ uint32_t mad_hi_next(uint32_t a, uint32_t b, uint32_t c) {
    return oz_chain((((uint64_t)a * b) >> 32) + c + oz_carry_flag);
}
#endif

}  // namespace ozlu
