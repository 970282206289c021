// Host builders of the kernels' small constant tables (tables.h).
#include "tables.h"

#include <string.h>

namespace ozlu {

void fill_conv(const DevTable& t, ConvTab& c) {
    memset(&c, 0, sizeof c);
    c.N = t.N; c.S = t.S; c.w = t.w; c.WX = t.WX;
    c.NW = (t.w + 1 + 31) / 32;
    for (int l = 0; l < t.N; ++l) {
        ConvMod& k = c.mod[l];
        const uint32_t m = (uint32_t)t.mod[l];
        uint32_t pw = 1 % m;  // 2^b mod m
        for (int b = 0; b <= 32 * CONV_WORDS; ++b) {
            if ((b & 7) == 0 && b < 32 * CONV_WORDS) k.p8[b >> 5] |= pw << (b & 31);
            if (b == t.w) k.wrapc = (m - pw) % m;
            if (b == 32 * c.NW) k.topc = (m - pw) % m;
            pw += pw;
            if (pw >= m) pw -= m;
        }
        k.m = m;
        k.magic = t.magic[l];
        k.half = m / 2;
        // binary16 of 1024 + half: exponent field 25, one unit per integer
        const uint32_t h = 0x6400u + k.half;
        k.h2 = h | (h << 16);
    }
}

}  // namespace ozlu
