// Host builders of the kernels' small constant tables (tables.h).
#include "tables.h"

#include <math.h>
#include <string.h>

namespace ozlu {

void fill_conv(const DevTable& t, ConvTab& c) {
    memset(&c, 0, sizeof c);
    c.N = t.N; c.S = t.S; c.w = t.w; c.WX = t.WX;
    c.NW = (t.w + 1 + 31) / 32;
    for (int l = 0; l < t.N; ++l) {
        ConvMod& k = c.mod[l];
        const uint32_t m = (uint32_t)t.mod[l];
        // x mod m for x < 2^24
        auto red = [&](uint32_t x) { return x - (uint32_t)(((uint64_t)x * t.magic[l]) >> 32) * m; };
        auto neg = [&](uint32_t x) { return x ? m - x : 0u; };
        uint32_t pw = 1 % m;  // 2^(8 b) mod m
        for (int b = 0; b <= 4 * CONV_WORDS; ++b) {
            if (b < 4 * CONV_WORDS) k.p8[b >> 2] |= pw << (8 * (b & 3));
            if (b == t.w >> 3) k.wrapc = neg(red(pw << (t.w & 7)));
            if (b == 4 * c.NW) k.topc = neg(pw);
            pw = red(pw << 8);
        }
        const uint32_t kneg = (1 + k.topc) % m;
        k.k4 = (k.wrapc << 8) | (kneg << 16) | ((kneg + m - k.wrapc) % m << 24);
        k.m = m;
        k.magic = t.magic[l];
        k.half = m / 2;
        // binary16 of 1024 + half: exponent field 25, one unit per integer
        const uint32_t h = 0x6400u + k.half;
        k.h2 = h | (h << 16);
    }
}

void fill_crt(const DevTable& t, int pint_bits, CrtTab& c) {
    memset(&c, 0, sizeof c);
    c.N = t.N; c.NT = (t.N + 2) / 3; c.WG = t.WG; c.G = t.G; c.w = t.w; c.g0 = t.g0;
    c.pint_bits = pint_bits;
    uint32_t mq[MAXTRI];  // products of triples, below 2^24
    for (int q = 0; q < c.NT; ++q) {
        mq[q] = 1;
        for (int l = 3 * q; l < 3 * q + 3 && l < t.N; ++l) mq[q] *= (uint32_t)t.mod[l];
        for (int l = 3 * q; l < 3 * q + 3 && l < t.N; ++l) c.coef[l] = mq[q] / (uint32_t)t.mod[l];
        c.inv[q] = 1.0f / (float)mq[q];
    }
    for (int q = 0; q < c.NT; ++q) {
        // P / m_q as the product of the other triples, modulo 2^(32 MAXWG)
        uint32_t* M = c.Mt[q];
        M[0] = 1;
        for (int j = 0; j < c.NT; ++j) {
            if (j == q) continue;
            uint64_t cy = 0;
            for (int k = 0; k < MAXWG; ++k) {
                cy += (uint64_t)M[k] * mq[j];
                M[k] = (uint32_t)cy;
                cy >>= 32;
            }
        }
    }
    uint64_t cy = 1;
    for (int k = 0; k < MAXWG; ++k) {
        cy += (uint32_t)~t.Plow[k];
        c.Pneg[k] = (uint32_t)cy;
        cy >>= 32;
    }
}

void fill_gemm(const DevTable& t, bool fp8, GemmTab& g) {
    memset(&g, 0, sizeof g);
    g.N = t.N; g.S = t.S; g.G = t.G; g.g0 = t.g0; g.NT = (t.N + 2) / 3;
    const int weight[2][3] = {{1, 0, 0}, {-16, 272, 17}};
    for (int l = 0; l < t.N; ++l) {
        GemmMod& k = g.mod[l];
        const int m = t.mod[l];
        k.m = (float)m;
        k.inv = 1.0f / k.m;
        k.invu = nextafterf(k.inv, 1.0f);
        double bound = 0.0;  // of |sum_p r_p y_p|, |r_p| <= 0.54 m + 1
        for (int p = 0; p < 3; ++p) {
            int y = (int)(((long long)weight[fp8 ? 1 : 0][p] * t.y[l]) % m);
            if (y < 0) y += m;
            if (y > m / 2) y -= m;
            k.y[p] = (float)y;
            bound += fabs((double)y) * (0.54 * m + 1.0);
        }
        k.off = (float)((long long)ceil(bound / m) * m);
        uint32_t mq = 1;
        for (int j = l / 3 * 3; j < l / 3 * 3 + 3 && j < t.N; ++j)
            if (j != l) mq *= (uint32_t)t.mod[j];
        k.coef = mq;
        g.ucorr[l / 3] -= 0x4b400000u * mq;
    }
}

}  // namespace ozlu
