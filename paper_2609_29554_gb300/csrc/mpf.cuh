// Multi-limb binary floating point on 32-bit integer limbs (device).
//
// value = (-1)^neg * m * 2^(e - 32 L), with m an L-word magnitude whose top
// bit is set (normalised), or zero (m = 0).  Every operation rounds its
// exact (or sticky-truncated) result to L words, round to nearest even.
// The arithmetic runs on the integer pipes (IMAD), which on GB300 issue
// about 40 times the binary64 FMA rate; the LU panel uses it for DD/TD/QD
// elements at 32 L >= 53 nc + 12 bits and converts to and from the
// expansion format (successive round-to-nearest on the way out).
#pragma once

#include <stdint.h>

#include "carry.cuh"
#include "mp_device.cuh"

namespace ozlu {

template <int L>
struct MPF {
    uint32_t m[L];
    int e;
    int neg;
};

template <int L>
__device__ __forceinline__ bool mpf_zero(const MPF<L>& a) {
    return a.m[L - 1] == 0;
}

template <int L>
__device__ __forceinline__ MPF<L> mpf_make_zero() {
    MPF<L> r;
#pragma unroll
    for (int i = 0; i < L; ++i) r.m[i] = 0;
    r.e = 0;
    r.neg = 0;
    return r;
}

// The rounding of a normalised W-word magnitude X 2^(ex - 32 W) to its top L
// words, to nearest even with a sticky for what lies below X: one carry chain
template <int L, int W>
__device__ __forceinline__ MPF<L> mpf_round_top(const uint32_t (&X)[W], int ex, int neg, bool sticky) {
    MPF<L> r;
    uint32_t up = 0;
    if (W > L) {
        uint32_t low = X[W - L - 1] & 0x7fffffffu;
#pragma unroll
        for (int i = 0; i < W - L - 1; ++i) low |= X[i];
        up = (X[W - L - 1] >> 31) & ((low != 0 || sticky) ? 1u : X[W - L] & 1u);
    }
    r.m[0] = add_first(X[W - L], up);
#pragma unroll
    for (int i = 1; i < L; ++i) r.m[i] = add_next(X[W - L + i], 0u);
    // X * 2^(ex - 32 W) with the top L words kept: m * 2^(ex - 32 L)
    r.e = ex;
    r.neg = neg;
    if (r.m[L - 1] == 0) {  // carried out: 1000...0
        r.m[L - 1] = 0x80000000u;
        r.e += 1;
    }
    return r;
}

// Round the W-word magnitude X (any leading zeros) to L words: normalise, keep
// the top 32 L bits, round to nearest even with a sticky.  `ex` is the exponent
// such that value = X * 2^(ex - 32 W).  Whole zero words at the top come only
// from a cancellation of 32 bits or more: they are shifted out one at a time.
template <int L, int W>
__device__ __forceinline__ MPF<L> mpf_round(uint32_t (&X)[W], int ex, int neg, bool sticky_in) {
    if (X[W - 1] == 0) {
        uint32_t any = 0;
#pragma unroll
        for (int i = 0; i < W - 1; ++i) any |= X[i];
        if (any == 0) return mpf_make_zero<L>();
        do {
#pragma unroll
            for (int i = W - 1; i > 0; --i) X[i] = X[i - 1];
            X[0] = 0;
            ex -= 32;
        } while (X[W - 1] == 0);
    }
    const int sh = __clz(X[W - 1]);
#pragma unroll
    for (int i = W - 1; i > 0; --i) X[i] = __funnelshift_l(X[i - 1], X[i], sh);
    X[0] <<= sh;
    return mpf_round_top<L, W>(X, ex - sh, neg, sticky_in);
}

// X += (neg ? -1 : 1) * mag * 2^pos (mod 2^(32 W)), pos >= 0, as one carry chain
template <int W>
__device__ __forceinline__ void mpf_acc(uint32_t (&X)[W], uint64_t mag, int pos, bool neg) {
    const int q = pos >> 5;
    const uint32_t m0 = (uint32_t)mag, m1 = (uint32_t)(mag >> 32), nm = neg ? 0xffffffffu : 0u;
    const uint32_t lo = __funnelshift_l(0u, m0, pos & 31), mid = __funnelshift_l(m0, m1, pos & 31),
                   hi = __funnelshift_l(m1, 0u, pos & 31);
    add_first(nm, nm & 1u);  // the flag: 1 for the complement
#pragma unroll
    for (int i = 0; i < W; ++i)
        X[i] = add_next(X[i], (i == q ? lo : i == q + 1 ? mid : i == q + 2 ? hi : 0u) ^ nm);
}

// from an expansion of N binary64 components (sticky-truncated to 32(L+2) bits,
// then rounded to L words).  The components are added with their sign relative
// to the first one's, so that the sum of a normalised expansion is positive.
template <int L, int N>
__device__ __forceinline__ MPF<L> mpf_from_exp(const double* x) {
    constexpr int W = L + 2;
    if (x[0] == 0.0) return mpf_make_zero<L>();
    const uint64_t b0 = (uint64_t)__double_as_longlong(x[0]);
    const int be = (int)((b0 >> 52) & 0x7ff);
    const int top = (be >= 1 && be <= 2046 ? be - 1022 : frexp_exp(x[0])) + 1;  // |value| < 2^top
    const int base = top - 32 * W;  // bit 0 of the window
    int neg = (int)(b0 >> 63);
    uint32_t X[W];
#pragma unroll
    for (int i = 0; i < W; ++i) X[i] = 0;
    bool sticky = false;
#pragma unroll
    for (int c = 0; c < N; ++c) {
        uint64_t mant;
        int e;
        bool ng;
        if (!decompose(x[c], mant, e, ng)) continue;
        int s = e - 53 - base;
        if (s < 0) {
            if (s <= -64) { sticky = true; continue; }
            if (mant & ((1ull << (-s)) - 1)) sticky = true;
            mant >>= -s;
            s = 0;
        }
        mpf_acc<W>(X, mant, s, ng != (neg != 0));
    }
    if (is_negative<W>(X)) {  // not normalised: the rest outweighs the first component
        negate<W>(X);
        neg ^= 1;
    }
    return mpf_round<L, W>(X, top, neg, sticky);
}

// q 2^e for q <= 2^53 (one rounding, for a subnormal result)
__device__ __forceinline__ double mpf_make_double(uint64_t q, int e, bool neg) {
    // 2^52 <= q <= 2^53 and a normal result: the biased exponent less one, plus
    // q with its top bit as it is
    if (q >> 52 && e >= -1073 && e <= 969)
        return __longlong_as_double((long long)((((uint64_t)(e + 1074) << 52) + q) | ((uint64_t)neg << 63)));
    const double x = scalbn((double)q, e);
    return neg ? -x : x;
}

// successive round-to-nearest-even into N binary64 components.  The magnitude
// is kept normalised: a component takes its top 53 bits, what is left of it (or
// what is missing, after a rounding up) moves to the top by 53 bits and its
// leading zeros.  Integer pipes only.
template <int L, int N>
__device__ __forceinline__ void mpf_to_exp(const MPF<L>& a, double* out) {
    uint32_t m[L];
#pragma unroll
    for (int i = 0; i < L; ++i) m[i] = a.m[i];
    bool neg = a.neg != 0;
    int e = a.e;  // |value| = m 2^(e - 32 L)
#pragma unroll
    for (int c = 0; c < N; ++c) {
        if (m[L - 1] == 0) {  // exhausted (or zero)
            out[c] = 0.0;
            continue;
        }
        const uint64_t hi = ((uint64_t)m[L - 1] << 32) | m[L - 2];
        uint64_t q = hi >> 11;
        const uint32_t low = m[L - 2] & 0x7ffu;
        uint32_t any = low & 0x3ffu;
#pragma unroll
        for (int i = 0; i < L - 2; ++i) any |= m[i];
        const bool up = (low & 0x400u) && (any || (q & 1));
        q += up;
        out[c] = mpf_make_double(q, e - 53, neg);
        if (c + 1 == N) break;
        // the rest r 2^-53, or 2^-53 - r after a rounding up: complemented
        // words below the 53 bits, moved up by 53 bits
        const uint32_t nm = up ? 0xffffffffu : 0u;
        uint32_t t[L];
        m[L - 1] = 0;
        m[L - 2] &= 0x7ffu;
        add_first(nm, nm & 1u);
#pragma unroll
        for (int i = 0; i < L - 1; ++i) t[i] = add_next(m[i] ^ nm, 0u);
        t[L - 2] &= 0x7ffu;
#pragma unroll
        for (int i = L - 1; i > 1; --i) m[i] = __funnelshift_l(t[i - 2], t[i - 1], 21);
        m[1] = t[0] << 21;
        m[0] = 0;
        e -= 53;
        neg ^= up;
        // leading zeros: whole words, then bits
#pragma unroll 1
        for (int w = 0; w < L - 1 && m[L - 1] == 0; ++w) {
#pragma unroll
            for (int i = L - 1; i > 0; --i) m[i] = m[i - 1];
            m[0] = 0;
            e -= 32;
        }
        const int sh = __clz(m[L - 1]) & 31;
#pragma unroll
        for (int i = L - 1; i > 0; --i) m[i] = __funnelshift_l(m[i - 1], m[i], sh);
        m[0] <<= sh;
        e -= sh;
    }
}

template <int L>
__device__ __forceinline__ MPF<L> mpf_neg(MPF<L> a) {
    a.neg ^= 1;
    return a;
}

// |a| vs |b|
template <int L>
__device__ __forceinline__ int mpf_abs_cmp(const MPF<L>& a, const MPF<L>& b) {
    const bool za = mpf_zero<L>(a), zb = mpf_zero<L>(b);
    if (za || zb) return za && zb ? 0 : (za ? -1 : 1);
    if (a.e != b.e) return a.e > b.e ? 1 : -1;
#pragma unroll
    for (int i = L - 1; i >= 0; --i)
        if (a.m[i] != b.m[i]) return a.m[i] > b.m[i] ? 1 : -1;
    return 0;
}

// Words K0 .. NA + NB - 1 of the product of an NA-word and an NB-word magnitude
// (exact for K0 = 0; else without the products below column K0, whose carry is
// under min(NA, NB) units of word K0).  Every 64-bit product a_i b_j is added at
// word i + j; those at even and at odd distance from K0 have an accumulator of
// their own, so that a row of each is one chain of wide multiply-adds on
// aligned word pairs (one instruction a product), and the two are added at the
// end.  7 x 7 words: 91 instructions and 315 cycles on one warp; the column sums
// of 32-bit halves that stood here before, 181 and 410.
template <int NA, int NB, int K0>
__device__ __forceinline__ void mul_words(const uint32_t (&a)[NA], const uint32_t (&b)[NB],
                                          uint32_t (&P)[NA + NB - K0]) {
    constexpr int W = NA + NB - K0;
    uint32_t E[W + 1], O[W + 1];  // O: word k + 1 at O[k]
#pragma unroll
    for (int k = 0; k <= W; ++k) {
        E[k] = 0;
        O[k] = 0;
    }
#pragma unroll
    for (int i = 0; i < NA; ++i) {
        int last = -1;
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int k = i + j - K0;
            if (k < 0 || (k & 1)) continue;
            E[k] = last < 0 ? mad_lo_first(a[i], b[j], E[k]) : mad_lo_next(a[i], b[j], E[k]);
            E[k + 1] = mad_hi_next(a[i], b[j], E[k + 1]);
            last = k;
        }
        // the word above a row's chain has only taken such carries so far
        if (last >= 0 && last + 2 < W) E[last + 2] = add_last(E[last + 2], 0u);
        last = -1;
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int k = i + j - K0;
            if (k < 0 || !(k & 1)) continue;
            O[k - 1] = last < 0 ? mad_lo_first(a[i], b[j], O[k - 1]) : mad_lo_next(a[i], b[j], O[k - 1]);
            O[k] = mad_hi_next(a[i], b[j], O[k]);
            last = k;
        }
        if (last >= 0 && last + 2 < W) O[last + 1] = add_last(O[last + 1], 0u);
    }
    P[0] = E[0];
    P[1] = add_first(E[1], O[0]);
#pragma unroll
    for (int k = 2; k < W; ++k) P[k] = add_next(E[k], O[k - 1]);
}

// a * b, rounded to L words
template <int L>
__device__ __forceinline__ MPF<L> mpf_mul(const MPF<L>& a, const MPF<L>& b) {
    if (mpf_zero<L>(a) || mpf_zero<L>(b)) return mpf_make_zero<L>();
    uint32_t P[2 * L];
    mul_words<L, L, 0>(a.m, b.m, P);
    // value = P * 2^((a.e + b.e) - 32 * 2L), P in [2^(64 L - 2), 2^(64 L)): one bit at most
    const int sh = P[2 * L - 1] >> 31 ? 0 : 1;
#pragma unroll
    for (int i = 2 * L - 1; i > 0; --i) P[i] = __funnelshift_l(P[i - 1], P[i], sh);
    P[0] <<= sh;
    return mpf_round_top<L, 2 * L>(P, a.e + b.e - sh, a.neg ^ b.neg, false);
}

// a + b, rounded to L words (guard words and a sticky keep it correctly rounded)
template <int L>
__device__ __forceinline__ MPF<L> mpf_add(const MPF<L>& a, const MPF<L>& b) {
    if (mpf_zero<L>(b)) return a;
    if (mpf_zero<L>(a)) return b;
    const bool swap = mpf_abs_cmp<L>(a, b) < 0;
    const MPF<L>& x = swap ? b : a;  // |x| >= |y|
    const MPF<L>& y = swap ? a : b;
    constexpr int W = L + 2;
    uint32_t X[W], Y[W];
    X[0] = 0;
    X[1] = 0;
    Y[0] = 0;
    Y[1] = 0;
#pragma unroll
    for (int i = 0; i < L; ++i) {
        X[i + 2] = x.m[i];
        Y[i + 2] = y.m[i];
    }
    // y shifted right by d = x.e - y.e bits (whole words by a logarithmic
    // shifter, then bits); sticky collects the bits shifted out
    const int d = x.e - y.e;
    bool sticky = false;
    if (d >= 32 * W) {
#pragma unroll
        for (int i = 0; i < W; ++i) Y[i] = 0;
        sticky = true;
    } else {
        const int q = d >> 5, r = d & 31;
#pragma unroll
        for (int s = 8; s >= 1; s >>= 1) {
            if (s < W) {
                const bool on = (q & s) != 0;
                uint32_t lost = 0;
#pragma unroll
                for (int i = 0; i < s; ++i) lost |= Y[i];
                sticky |= on && lost != 0;
#pragma unroll
                for (int i = 0; i < W; ++i) Y[i] = on ? (i + s < W ? Y[i + s] : 0u) : Y[i];
            }
        }
        sticky |= r != 0 && (Y[0] & ((1u << r) - 1u)) != 0;
#pragma unroll
        for (int i = 0; i < W - 1; ++i) Y[i] = __funnelshift_r(Y[i], Y[i + 1], r);
        Y[W - 1] >>= r;
    }
    if (x.neg == y.neg) {
        uint64_t c = 0;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const uint64_t s = (uint64_t)X[i] + Y[i] + c;
            X[i] = (uint32_t)s;
            c = s >> 32;
        }
        // carry out of the window: shift right one bit, keep the lost bit
        if (c) {
            sticky |= (X[0] & 1u) != 0;
#pragma unroll
            for (int i = 0; i < W - 1; ++i) X[i] = (X[i] >> 1) | (X[i + 1] << 31);
            X[W - 1] = (X[W - 1] >> 1) | 0x80000000u;
            return mpf_round<L, W>(X, x.e + 1, x.neg, sticky);
        }
        return mpf_round<L, W>(X, x.e, x.neg, sticky);
    }
    // |x| >= |y|: the exact difference is X - Y - delta with 0 <= delta < 1
    // unit of the window (the bits of y below it); X - Y - 1 plus a set sticky
    // stands for it whenever delta > 0
    uint64_t brw = sticky ? 1u : 0u;
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const uint64_t s = (uint64_t)X[i] - Y[i] - brw;
        X[i] = (uint32_t)s;
        brw = (s >> 63) & 1u;
    }
    return mpf_round<L, W>(X, x.e, x.neg, sticky);
}

// c - a b with one rounding: the product's top L + 2 words (from the columns
// that reach them and one guard column; what is left out is under 2^-28 of
// the lowest window word) meet c in an (L + 2)-word window, the lower words
// counting as a set sticky.  The result is the correctly rounded c - a b unless
// the exact value lies within about 2^-58 of a unit of its last word from a
// rounding boundary.  Written for a short dependent chain and few
// instructions, since the LU's panels and triangular solves run it on one warp
// or two per scheduler: chains on the carry flag throughout, the alignment by
// a loop over whole words (the exponents mostly lie within a word or two) and one
// funnel shift, addition and subtraction as one chain on B or its complement.
// L = 7: 724 cycles on one warp, 96 SM cycles a warp with 16 of them; the QD
// triangular solves of the n = 4096 LU went from 14.3 to 10.3 ms with it.
template <int L>
__device__ __forceinline__ MPF<L> mpf_fms(const MPF<L>& c, const MPF<L>& a, const MPF<L>& b) {
    static_assert(L >= 4, "two guard words below the product window");
    constexpr int W = L + 2;
    if (mpf_zero<L>(a) || mpf_zero<L>(b)) return c;
    uint32_t G[W + 1];
    mul_words<L, L, L - 3>(a.m, b.m, G);
    // a b ~ P 2^(ep - 32 W), P the top W words of G, normalised (the top bit may be clear)
    const int up1 = G[W] >> 31 ? 0 : 1;
    uint32_t P[W];
#pragma unroll
    for (int i = 0; i < W; ++i) P[i] = __funnelshift_l(G[i], G[i + 1], up1);
    const int ep = a.e + b.e - up1;
    const int pn = a.neg ^ b.neg ^ 1;
    if (mpf_zero<L>(c)) return mpf_round_top<L, W>(P, ep, pn, true);
    // A: the operand of the larger exponent (c on a tie), B the other
    const bool swap = ep > c.e;
    uint32_t A[W], B[W];
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const uint32_t cw = i < 2 ? 0u : c.m[i < 2 ? 0 : i - 2];
        A[i] = swap ? P[i] : cw;
        B[i] = swap ? cw : P[i];
    }
    const int ea = swap ? ep : c.e;
    int an = swap ? pn : c.neg;
    int d = swap ? ep - c.e : c.e - ep;
    // B >>= d; the bits shifted out and, where B is the product, its words left
    // out make the sticky
    bool sticky = !swap;
    if (d >= 32 * W) {
        sticky = true;
#pragma unroll
        for (int i = 0; i < W; ++i) B[i] = 0;
    } else {
        uint32_t lost = 0;
        for (; d >= 32; d -= 32) {
            lost |= B[0];
#pragma unroll
            for (int i = 0; i < W - 1; ++i) B[i] = B[i + 1];
            B[W - 1] = 0;
        }
        lost |= __funnelshift_r(0u, B[0], d);
        sticky |= lost != 0;
#pragma unroll
        for (int i = 0; i < W - 1; ++i) B[i] = __funnelshift_r(B[i], B[i + 1], d);
        B[W - 1] >>= d;
    }
    // A + B, or A - B - delta with 0 < delta < 1 unit of the window where the
    // sticky is set: A - B - 1 plus a set sticky stands for it
    const uint32_t f = c.neg != pn ? 0xffffffffu : 0u;
    add_first(f, f & (sticky ? 0u : 1u));  // the flag: set for an exact difference
#pragma unroll
    for (int i = 0; i < W; ++i) A[i] = add_next(A[i], B[i] ^ f);
    const uint32_t cy = add_last(0u, 0u);
    if (f == 0) {
        if (cy) {
            sticky |= (A[0] & 1u) != 0;
#pragma unroll
            for (int i = 0; i < W - 1; ++i) A[i] = __funnelshift_r(A[i], A[i + 1], 1);
            A[W - 1] = (A[W - 1] >> 1) | 0x80000000u;
            return mpf_round_top<L, W>(A, ea + 1, an, sticky);
        }
    } else if (!cy) {
        // A < B + delta (equal exponents): B - A of the other sign; zero for an
        // exact cancellation such as c = a b
#pragma unroll
        for (int i = 0; i < W; ++i) A[i] = ~A[i];
        an ^= 1;
        sticky = false;
    }
    return mpf_round<L, W>(A, ea, an, sticky);
}

// An out-of-line copy of the fused multiply-subtract.  A kernel whose warps run
// several at once on different code paths (the LU panel) then keeps one copy in the
// instruction cache instead of one per call site.  Operands and result go by
// value, in registers.
template <int L>
__device__ __noinline__ MPF<L> mpf_fms_oolv(MPF<L> c, MPF<L> a, MPF<L> b) {
    return mpf_fms<L>(c, a, b);
}

template <int L>
__device__ __forceinline__ MPF<L> mpf_from_double(double v) {
    return mpf_from_exp<L, 1>(&v);
}

template <int L>
__device__ __forceinline__ MPF<L> mpf_one() {
    MPF<L> r = mpf_make_zero<L>();
    r.m[L - 1] = 0x80000000u;
    r.e = 1;
    return r;
}

// (top word of |a|)^2: a^2 to about 30 bits, positive (integer pipes only)
template <int L>
__device__ __forceinline__ MPF<L> mpf_top_square(const MPF<L>& a) {
    MPF<L> r = mpf_make_zero<L>();
    if (mpf_zero<L>(a)) return r;
    // |a| ~ m_top 2^(a.e - 32), a^2 ~ q 2^(2 a.e - 64) with q = m_top^2 >= 2^62
    uint64_t q = (uint64_t)a.m[L - 1] * a.m[L - 1];
    int e = 2 * a.e;
    if (!(q >> 63)) {
        q <<= 1;
        e -= 1;
    }
    r.m[L - 1] = (uint32_t)(q >> 32);
    r.m[L - 2] = (uint32_t)q;
    r.e = e;
    return r;
}

// the same value with K < L words (low words zero)
template <int L, int K>
__device__ __forceinline__ MPF<L> mpf_widen(const MPF<K>& a) {
    MPF<L> r;
#pragma unroll
    for (int i = 0; i < L - K; ++i) r.m[i] = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) r.m[L - K + i] = a.m[i];
    r.e = a.e;
    r.neg = a.neg;
    return r;
}

// 1 / f to about 60 bits for f = T 2^-64 + (lower bits) in [1/2, 1),
// T in [2^63, 2^64): a binary32 reciprocal of the top 24 bits (relative error
// below 2^-22), then two Newton steps r <- r + r e, e = 1 - T r 2^-64, in
// 62-bit fixed point R = r 2^62 with 64 x 64-bit integer products (error
// about 2^-44, then about 2^-61, the limit of R and of T).  No binary64.
__device__ __forceinline__ MPF<4> mpf_recip_seed(uint64_t T) {
    const float tf = (float)(uint32_t)(T >> 40);  // [2^23, 2^24), exact
    const uint32_t bits = __float_as_uint(__frcp_rn(tf));
    const int ex = (int)((bits >> 23) & 0xffu) - 127;  // 1 / tf in (2^-24, 2^-23]: -24 or -23
    uint64_t R = (uint64_t)((bits & 0x7fffffu) | 0x800000u) << (ex + 63);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        // E = 2^126 - T R (signed 128-bit), e = E 2^-126; |E| < 2^104, then < 2^82,
        // so E >> sh fits in 63 bits
        const uint64_t lo = T * R, hi = __umul64hi(T, R);
        const uint64_t elo = 0ull - lo;
        const uint64_t ehi = (1ull << 62) - hi - (lo != 0ull ? 1ull : 0ull);
        const int sh = s == 0 ? 41 : 20;
        const int64_t es = (int64_t)((ehi << (64 - sh)) | (elo >> sh));
        // R e = R es 2^(sh - 126) = umulhi(R, |es|) 2^(sh - 62)
        const uint64_t d = __umul64hi(R, es < 0 ? (uint64_t)(-es) : (uint64_t)es) >> (62 - sh);
        R = es < 0 ? R - d : R + d;
    }
    // r = R 2^-62 as a 4-word float: R normalised into the top two words
    const int z = __clzll((long long)R);
    const uint64_t M = R << z;
    MPF<4> r;
    r.m[3] = (uint32_t)(M >> 32);
    r.m[2] = (uint32_t)M;
    r.m[1] = 0;
    r.m[0] = 0;
    r.e = 2 - z;
    r.neg = 0;
    return r;
}

// 1 / f for f = F 2^(-32 L) in (1/2, 1), L <= 7, in fixed point: R words with
// r = R 2^(1 - 32 (L + 1)) in (1, 2), r < 1 / f, 1 - f r < 2^-(32 L + 28).
// Newton steps r <- r + r e, e = 1 - f r, whose result (1 - e^2) / f stays below
// 1 / f (with the e^2 of the last one added, L = 7, (1 - e^3) / f); each uses only
// the words of f and of e that its precision needs, so that the alignments are
// fixed and nothing is normalised.  On values:
//   r0  binary32 reciprocal of the top 24 bits plus one       e < 2^-21
//   r1  32-bit f (plus one unit), one step in 64 bits          e < 2^-30
//   r2  64-bit f (plus one unit), one step                     e < 2^-59
//   r3  four words of f (plus one unit), two of r              e < 2^-117
//   r4  all of f, four words of r
// 62 wide multiply-adds for L = 7, against four fused multiply-subtracts of
// general floats before (3413 cycles on one thread with the present ones; 783 now).
template <int L>
__device__ __forceinline__ void recip_words(const uint32_t (&F)[L], uint32_t (&R)[L + 1]) {
    const uint32_t t32 = F[L - 1];
    const uint64_t T = ((uint64_t)t32 << 32) | F[L - 2];
    // r0 2^30, a binary32 unit below
    const uint32_t fb = __float_as_uint(__frcp_rn((float)((t32 >> 8) + 1)));
    // (1 / (t + 1) in [2^-24, 2^-23): exponent field 103; 2^-24 itself only for t + 1 = 2^24)
    const uint32_t R0 = (((fb & 0x7fffffu) | 0x800000u) << 7) - 128u;
    // r1 2^62
    const uint64_t E1 = (1ull << 62) - ((uint64_t)R0 * t32 + R0);
    const uint64_t R1 = ((uint64_t)R0 << 32) + (((uint64_t)R0 * (uint32_t)(E1 >> 10)) >> 20);
    // r2 2^62: E2 = 2^126 - (T + 1) R1
    const uint64_t plo = T * R1, lo2 = plo + R1;
    const uint64_t hi2 = __umul64hi(T, R1) + (lo2 < plo ? 1ull : 0ull);
    const uint64_t elo = 0ull - lo2, ehi = (1ull << 62) - hi2 - (lo2 != 0ull ? 1ull : 0ull);
    const uint64_t R2 = R1 + (__umul64hi(R1, (ehi << 31) | (elo >> 33)) >> 29);
    // r3 2^127 in four words: E3 = 2^191 - (F4 + 1) G, G = r2 2^63
    const uint32_t G[2] = {(uint32_t)(R2 << 1), (uint32_t)(R2 >> 31)};
    uint32_t F4[4], P3[6], R3[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) F4[i] = F[L - 4 + i];
    mul_words<4, 2, 0>(F4, G, P3);
    P3[0] = add_first(P3[0], G[0]);
    P3[1] = add_next(P3[1], G[1]);
#pragma unroll
    for (int i = 2; i < 6; ++i) P3[i] = add_next(P3[i], 0u);
    {
        // -P3 = ~P3 + 1; E3 < 2^132: words 2 .. 4
        add_first(~P3[0], 1u);
        add_next(~P3[1], 0u);
        uint32_t E3[3], Q[5];
#pragma unroll
        for (int i = 0; i < 3; ++i) E3[i] = add_next(~P3[i + 2], 0u);
        mul_words<3, 2, 0>(E3, G, Q);
        // r3 2^127 = G 2^64 + (G E3) 2^-63
        R3[0] = __funnelshift_r(Q[1], Q[2], 31);
        R3[1] = __funnelshift_r(Q[2], Q[3], 31);
        const uint32_t q2 = __funnelshift_r(Q[3], Q[4], 31);
        R3[2] = add_first(G[0], q2);
        R3[3] = add_last(G[1], Q[4] >> 31);
    }
    // r4: E4 = 2^(32 L + 127) - F R3 < 2^(32 L + 12): words 0 .. L; its top NE
    // words times R3
    constexpr int NE = L - 2, WP = L + 4;
    uint32_t P4[WP], E4[NE], Q[NE + 4];
    mul_words<L, 4, 0>(F, R3, P4);
    add_first(~P4[0], 1u);
#pragma unroll
    for (int i = 1; i < L + 1 - NE; ++i) add_next(~P4[i], 0u);
#pragma unroll
    for (int i = 0; i < NE; ++i) E4[i] = add_next(~P4[L + 1 - NE + i], 0u);
    if (L >= 7) {
        // the step's third-order term e^2 (2^-234 at most, below the words kept for
        // L <= 6): e = t 2^-147 from the top 32 bits, e^2 in units of E4's word 0
        const uint32_t t = __funnelshift_r(E4[NE - 2], E4[NE - 1], 12);
        E4[0] = add_first(E4[0], __umulhi(t, t) >> (L >= 7 ? 231 - 32 * L : 0));
#pragma unroll
        for (int i = 1; i < NE; ++i) E4[i] = add_next(E4[i], 0u);
    }
    mul_words<NE, 4, 0>(E4, R3, Q);
    // r 2^(32 L + 31) = R3 2^(32 L - 96) + R3 E4 2^-223, E4 here without its low
    // L + 1 - NE = 3 words: (R3 E4) 2^-127, words from bit 127 on
    uint32_t q[L + 1];
#pragma unroll
    for (int i = 0; i < L + 1; ++i)
        q[i] = i + 3 < NE + 4 ? __funnelshift_r(Q[i + 3 < NE + 4 ? i + 3 : 0], i + 4 < NE + 4 ? Q[i + 4 < NE + 4 ? i + 4 : 0] : 0u, 31) : 0u;
    R[0] = L - 3 <= 0 ? add_first(q[0], R3[0]) : q[0];
#pragma unroll
    for (int i = 1; i < L + 1; ++i) {
        if (i < L - 3) R[i] = q[i];
        else if (i == L - 3) R[i] = add_first(q[i], R3[0]);
        else R[i] = add_next(q[i], R3[i - (L - 3) < 4 ? i - (L - 3) : 0]);
    }
}

// the general-float steps of mpf_recip for L >= 8
template <int L>
__device__ __forceinline__ MPF<L> mpf_recip_long(const MPF<L>& b) {
    MPF<4> r4 = mpf_recip_seed(((uint64_t)b.m[L - 1] << 32) | b.m[L - 2]);
    MPF<4> f4;
#pragma unroll
    for (int i = 0; i < 4; ++i) f4.m[i] = b.m[L - 4 + i];
    f4.e = 0;
    f4.neg = 0;
    {
        MPF<4> t4 = mpf_fms<4>(mpf_one<4>(), f4, r4);
        r4 = mpf_fms<4>(r4, r4, mpf_neg<4>(t4));
    }
    MPF<L> r = mpf_widen<L, 4>(r4);
    {
        MPF<L> f = b;
        f.neg = 0;
        f.e = 0;
        MPF<L> t = mpf_fms<L>(mpf_one<L>(), f, r);
        t = mpf_add<L>(t, mpf_top_square<L>(t));
        r = mpf_fms<L>(r, r, mpf_neg<L>(t));
        for (int prec = 360; prec < 32 * L + 8; prec *= 2) {
            t = mpf_fms<L>(mpf_one<L>(), f, r);
            r = mpf_fms<L>(r, r, mpf_neg<L>(t));
        }
    }
    r.e -= b.e;
    r.neg = b.neg;
    return r;
}

// 1 / b on the mantissa f = |b| 2^-e in [1/2, 1), the exponent applied last.
// L <= 7 takes the fixed-point steps above; a power of two is exact.  Longer
// formats work on general floats: from the seed r (above), the residual
// e = 1 - f r of one fused multiply-subtract (a single rounding) gives
// r = (1 - e) / f exactly, so
//   r (1 + e)       = (1 - e^2) / f   (second order),
//   r (1 + e + e^2) = (1 - e^3) / f   (third order, e^2 from the top word of e),
// each formed as r + r t by one more fused multiply-subtract: a 4-word step of
// second order (about 120 bits) on the top 128 bits of f, then one L-word step of
// third order (about 360 bits) and second-order steps beyond.  Everything runs
// on the integer pipes apart from one binary32 reciprocal.
template <int L>
__device__ __forceinline__ MPF<L> mpf_recip(const MPF<L>& b) {
    static_assert(L >= 4, "a 4-word first step");
    if constexpr (L <= 7) {
        uint32_t low = b.m[L - 1] ^ 0x80000000u;
#pragma unroll
        for (int i = 0; i < L - 1; ++i) low |= b.m[i];
        if (low == 0) {  // 1 / 2^(e - 1) = 2^(1 - e)
            MPF<L> r = mpf_one<L>();
            r.e = 2 - b.e;
            r.neg = b.neg;
            return r;
        }
        uint32_t R[L + 1];
        recip_words<L>(b.m, R);
        return mpf_round_top<L, L + 1>(R, 1 - b.e, b.neg, true);
    } else {
        return mpf_recip_long<L>(b);
    }
}

}  // namespace ozlu
