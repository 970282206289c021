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
    // p-bit digits sgn (D - wrap 2^w), D replaced by its complement where
    // negative: byte neg 2 + wrap is the correction {0, -2^w, 1 - 2^(32 NW),
    // 1 - 2^(32 NW) + 2^w} mod m
    uint32_t k4;
    uint32_t pad_;
};

struct ConvTab {
    int N, S, w, NW, WX;  // NW: words of a digit, ceil((w + 1) / 32); WX: words of X
    int pad_[3];
    ConvMod mod[MAXMOD];
};

// CRT of one digit group by triples of moduli.  With m_q = m_a m_b m_c,
//   u_q = t_a m_b m_c + t_b m_a m_c + t_c m_a m_b   (< 3 * 255^3 < 2^26)
// the sum of Eq. (11) is S_g = sum_q u_q (P / m_q) - round(F) P with
// F = sum_q u_q / m_q: a third of the word products, and every sum of up to 18
// products u_q * word (and round(F) times a word of P) stays below 2^62.  A last group of one or two moduli
// leaves the others out (coefficient 0).
constexpr int MAXTRI = 18;  // the 54 moduli <= 255

struct CrtTab {
    int N, NT, WG, G, w, g0;
    int pint_bits;                 // |P_int| < 2^pint_bits
    int pad_;
    uint32_t coef[3 * MAXTRI];     // m_q / m_l
    float inv[MAXTRI];             // 1 / m_q
    uint32_t Mt[MAXTRI][MAXWG];    // P / m_q mod 2^(32 WG)
    uint32_t Pneg[MAXWG];          // -P mod 2^(32 WG)
};

// One modulus of the tensor-core epilogue, which works in binary32 on exact
// integers: t = (C y) mod m from C = sum_p weight_p C_p (FP16: one product;
// FP8: the planes of Eq. (15), C = -16 P00 + 17 Pss + 272 P11 in the order
// d0, d1, d0 + d1).
struct GemmMod {
    float m, inv;     // inv = 1 / m to nearest
    float invu;       // the next binary32 above it
    float y[3];       // (weight_p y_l) mod m, centered
    float off;        // a multiple of m that makes sum_p r_p y_p + off >= 0
    uint32_t coef;    // m_q / m of the modulus' triple (CrtTab)
};

struct GemmTab {
    int N, S, G, g0, NT, pad_[3];
    GemmMod mod[MAXMOD];
    uint32_t ucorr[MAXTRI];  // -(bits of 1.5 2^23) sum of the triple's coef
};

void fill_gemm(const DevTable& t, bool fp8, GemmTab& g);

// from the plan's table; pint_bits as the plan counts them
void fill_crt(const DevTable& t, int pint_bits, CrtTab& c);

// from the plan's table (the moduli <= 255 of the INT8, FP8 and FP16 back-ends)
void fill_conv(const DevTable& t, ConvTab& c);

}  // namespace ozlu
