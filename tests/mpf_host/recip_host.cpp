// The fixed-point reciprocal of the device floats (recip_words of csrc/mpf.cuh) on
// the CPU: per line L, the words of f and those of the result, top word first.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#define __device__
#define __forceinline__ inline
#define __noinline__
static inline int __clz(uint32_t x) { return x ? __builtin_clz(x) : 32; }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline long long __double_as_longlong(double d) { long long r; memcpy(&r, &d, 8); return r; }
static inline double __longlong_as_double(long long x) { double r; memcpy(&r, &x, 8); return r; }
static inline uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static inline float __frcp_rn(float x) { volatile float one = 1.0f; return one / x; }
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) {
    s &= 31;
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
static inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) {
    s &= 31;
    return s ? (lo >> s) | (hi << (32 - s)) : lo;
}

#include "mpf.cuh"

using namespace ozlu;

template <int L>
static void run(int n) {
    std::mt19937_64 g(L);
    for (int i = 0; i < n; ++i) {
        uint32_t F[L], R[L + 1];
        for (int k = 0; k < L; ++k) F[k] = (uint32_t)g();
        if (i % 8 == 1) for (int k = 0; k < L; ++k) F[k] = 0xffffffffu;                       // next to 1
        if (i % 8 == 2) for (int k = 1; k < L; ++k) F[k] = 0;                                 // next to 1/2
        if (i % 8 == 3) F[L - 1] = (uint32_t)(g() << 8) | 0xffu, F[L - 2] = 0xffffffffu;      // the seed's worst
        if (i % 8 == 4) F[L - 1] = (uint32_t)(g() % 4096), F[L - 1] |= 0x80000000u;
        F[0] |= 1u;
        F[L - 1] |= 0x80000000u;
        recip_words<L>(F, R);
        printf("%d ", L);
        for (int k = L - 1; k >= 0; --k) printf("%08x", F[k]);
        printf(" ");
        for (int k = L; k >= 0; --k) printf("%08x", R[k]);
        printf("\n");
    }
}

int main(int argc, char** argv) {
    const int n = argc > 1 ? atoi(argv[1]) : 1000;
    run<4>(n);
    run<6>(n);
    run<7>(n);
    return 0;
}
