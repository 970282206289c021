// Small constant tables of the kernels, built on the host from a plan's
// DevTable and passed by value.  Each kernel gets only what it reads: a
// launch copies its parameters, and the full DevTable is 9.6 KB.
#pragma once

#include <stdint.h>

#include "ozlu_internal.h"

namespace ozlu {

constexpr int CONV_WORDS = 8;  // 32-bit words of one balanced digit (w + 1 <= 256 bits)

// One modulus of the conversion, 64 bytes.  A digit is kept as an unsigned
// value of NW words less a power of two (wrapped lower digits: 2^w; a negative
// top digit: 2^(32 NW), its two's complement), so its centered residue is
//   (half + [wrapped] minus_pow + sum_j byte_j (2^(8 j) mod m)) mod m - half,
// half = floor(m / 2).
struct ConvMod {
    uint32_t p8[CONV_WORDS];  // word k: the bytes 2^(32 k + 8 j) mod m, j = 0..3
    uint32_t m, magic;        // ceil(2^32 / m): exact floor(x / m) for x < 2^24
    uint32_t half;
    uint32_t wrapc;           // -2^w mod m
    uint32_t topc;            // -2^(32 NW) mod m
    uint32_t h2;              // binary16 pair (1024 + half, 1024 + half)
    uint32_t pad_[2];
};

struct ConvTab {
    int N, S, w, NW, WX;  // NW: words of a digit, ceil((w + 1) / 32); WX: words of X
    int pad_[3];
    ConvMod mod[MAXMOD];
};

// from the plan's table (the moduli <= 255 of the INT8, FP8 and FP16 back-ends)
void fill_conv(const DevTable& t, ConvTab& c);

}  // namespace ozlu
