// Device code shared by the conversions of expansions and of p-bit numbers: the
// residues of E consecutive plane positions, packed and stored at once.
#pragma once

#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <string.h>

#include "tables.h"

namespace ozlu {

// balanced base-17 digits of Eq. (15) of two centered residues (binary16
// pair): r = 17 d1 + d0, d1 = round(r / 17) (no ties: 17 is odd); 1536 is the
// rounding constant of integers in binary16, every step is exact
__device__ __forceinline__ void base17(__half2 c, uint32_t& e0, uint32_t& e1, uint32_t& es) {
    const __half2 big = __floats2half2_rn(1536.0f, 1536.0f);
    const __half2 d1 = __hsub2(__hfma2(c, __floats2half2_rn(1.0f / 17.0f, 1.0f / 17.0f), big), big);
    const __half2 d0 = __hfma2(d1, __floats2half2_rn(-17.0f, -17.0f), c);
    const __half2 ds = __hadd2(d0, d1);
    e0 = __nv_cvt_halfraw2_to_fp8x2(d0, __NV_SATFINITE, __NV_E4M3);
    e1 = __nv_cvt_halfraw2_to_fp8x2(d1, __NV_SATFINITE, __NV_E4M3);
    es = __nv_cvt_halfraw2_to_fp8x2(ds, __NV_SATFINITE, __NV_E4M3);
}

__device__ __forceinline__ __half2 as_half2(uint32_t v) {
    __half2 h;
    memcpy(&h, &v, 4);
    return h;
}

__device__ __forceinline__ uint32_t as_u32(__half2 h) {
    uint32_t v;
    memcpy(&v, &h, 4);
    return v;
}

// centered residue + half of the digit in D (ConvMod); acc starts as half plus
// the digit's power-of-two correction
template <int NW>
__device__ __forceinline__ uint32_t conv_residue(const uint32_t (&D)[NW], const ConvMod& M, uint32_t acc) {
#pragma unroll
    for (int i = 0; i < NW; ++i) acc = __dp4a(D[i], M.p8[i], acc);
    return acc - __umulhi(acc, M.magic) * M.m;
}

// res[e]: centered residue + half of position off + e, to plane(s) `index`:
// MODE 0 int8, 1 the three E4M3 digit planes 3 index + 0..2, 2 binary16
template <int MODE, int E>
__device__ __forceinline__ void store_residues(void* planes, size_t index, size_t plane, size_t off, const ConvMod& M,
                                               const uint32_t (&res)[E]) {
    const size_t at = index * (MODE == 1 ? 3 : 1) * plane + off;
    if (MODE == 0) {
        int8_t* dst = (int8_t*)planes + at;
        if (E == 4) {
            const uint32_t lo = __byte_perm(res[0] - M.half, res[E > 1 ? 1 : 0] - M.half, 0x0040);
            const uint32_t hi = __byte_perm(res[E > 2 ? 2 : 0] - M.half, res[E > 3 ? 3 : 0] - M.half, 0x0040);
            *(uint32_t*)dst = __byte_perm(lo, hi, 0x5410);
        } else {
            *dst = (int8_t)(res[0] - M.half);
        }
    } else {
        // binary16 of 1024 + res is 0x6400 + res; less 1024 + half, exact
        uint32_t c2[E > 2 ? 2 : 1];
#pragma unroll
        for (int q = 0; q < (E > 2 ? 2 : 1); ++q)
            c2[q] = as_u32(__hsub2(as_half2(res[E > 1 ? 2 * q : 0] + (E > 1 ? res[E > 1 ? 2 * q + 1 : 0] << 16 : 0u) +
                                            0x64006400u),
                                   as_half2(M.h2)));
        if (MODE == 2) {
            __half* dst = (__half*)planes + at;
            if (E == 4) *(uint2*)dst = make_uint2(c2[0], c2[E > 2 ? 1 : 0]);
            else *(uint16_t*)dst = (uint16_t)c2[0];
        } else {
            uint32_t f[3], g[3] = {0, 0, 0};
            base17(as_half2(c2[0]), f[0], f[1], f[2]);
            if (E == 4) base17(as_half2(c2[E > 2 ? 1 : 0]), g[0], g[1], g[2]);
            uint8_t* dst = (uint8_t*)planes + at;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (E == 4) *(uint32_t*)(dst + q * plane) = f[q] | (g[q] << 16);
                else dst[q * plane] = (uint8_t)f[q];
            }
        }
    }
}

}  // namespace ozlu
