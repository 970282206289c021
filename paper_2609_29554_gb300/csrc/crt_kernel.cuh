// CRT kernel of the byte-modulus back-ends (see crt.cu), a template over the
// layout of the t values; crt_bytes.cu and crt_packed.cu instantiate one each
// (two translation units compile side by side).
#pragma once

#include "launch.cuh"
#include "carry.cuh"
#include "mp_device.cuh"
#include "ozlu_internal.h"
#include "tables.h"

namespace ozlu {

struct CrtArgs {
    const void* T;
    const int* mu;
    const int* nu;
    double* C;
    long long ldc, mn;
    int m, nc, alpha, beta;
    int vec;  // elements of 2 or 4 components on a 16-byte boundary: 16-byte loads and stores
};

void launch_crt_bytes(const CrtArgs& a, const CrtTab& tab, cudaStream_t s);
void launch_crt_packed(const CrtArgs& a, const CrtTab& tab, cudaStream_t s);

namespace {

// ---------------------------------------------------------------------------
// The kernel of the byte-modulus back-ends.  One thread per output, everything
// in registers: the window X is NW words (a template parameter, the plan's
// P_int and 30 bits or more to spare for the old C), so that shifts by the
// plan's w are uniform word moves and funnel shifts, and the only shift by an
// amount of the thread's own is the normalisation.  It is bound by integer
// issue.  Per output of a QD update (S = 2, 32 moduli, K = 256): 11 triples x 8
// words x 2 groups of products, the old C's four components placed in the
// window, and one normalised residual per output component, whose 53 bits,
// round bit and sticky then sit at fixed places.
// 3840 x 3840, beta = 1, S = 2: 1058 us from packed words; the former kernel (one
// modulus at a time, the window in shared memory, run-time loops) 2080 us.
//
// An old C whose exponent lies too far above the grid for NW words takes the
// out-of-line copy with WACC words, which also raises the grid (WINDOW_BITS).
constexpr int CT = 128;  // threads per block
// Blocks per SM the registers are limited for.  The t loads' latency wants warps
// more than the window wants registers: packed, QD 3840 x 3840 update, 5 / 6 / 7
// / 8 blocks 1299 / 1158 / 1097 / 1058 us; bytes (twelve loads in flight per
// step), TD 1777 x 611, 78 / 72 / 76 / 80 us.
template <int NW, bool PACK>
constexpr int min_blocks() { return PACK && NW <= 13 ? 8 : 6; }

// X <<= 32 Q + r
template <int NW, int Q>
__device__ __forceinline__ void shl_words(uint32_t (&X)[NW], int r) {
#pragma unroll
    for (int i = NW - 1; i >= 0; --i)
        X[i] = i < Q ? 0u : __funnelshift_l(i > Q ? X[i > Q ? i - Q - 1 : 0] : 0u, X[i >= Q ? i - Q : 0], r);
}

// X <<= w (uniform w < 256)
template <int NW>
__device__ __forceinline__ void shl_uniform(uint32_t (&X)[NW], int w) {
    const int r = w & 31;
    switch (w >> 5) {
        case 0: shl_words<NW, 0>(X, r); break;
        case 1: shl_words<NW, 1>(X, r); break;
        case 2: shl_words<NW, 2>(X, r); break;
        case 3: shl_words<NW, 3>(X, r); break;
        case 4: shl_words<NW, 4>(X, r); break;
        case 5: shl_words<NW, 5>(X, r); break;
        case 6: shl_words<NW, 6>(X, r); break;
        default: shl_words<NW, 7>(X, r); break;
    }
}

// X = -X where neg
template <int NW>
__device__ __forceinline__ void negate_if(uint32_t (&X)[NW], bool neg) {
    const uint32_t f = neg ? 0xffffffffu : 0u;
    X[0] = add_first(X[0] ^ f, neg ? 1u : 0u);
#pragma unroll
    for (int i = 1; i < NW; ++i) X[i] = add_next(X[i] ^ f, 0u);
}

// The u_q of triples [4 b, 4 b + 4) of digit group gi, output e: words of the
// packed layout T[gi][q][e], or formed by triple() from the bytes T[gi][l][e]
// (zero past the last modulus; the table's rows there are zero).
template <bool PACK>
struct Fetch {
    uint32_t t[PACK ? 4 : 12];
    __device__ __forceinline__ void load(const CrtArgs& a, const CrtTab& tab, long long e, int gi, int b) {
        if (PACK) {
            const uint32_t* tp = (const uint32_t*)a.T + ((long long)gi * tab.NT + 4 * b) * a.mn + e;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                t[i] = 4 * b + i < tab.NT ? *tp : 0u;
                tp += a.mn;
            }
        } else {
            const uint8_t* tp = (const uint8_t*)a.T + ((long long)gi * tab.N + 12 * b) * a.mn + e;
#pragma unroll
            for (int i = 0; i < (PACK ? 4 : 12); ++i) {
                t[i] = 12 * b + i < tab.N ? (uint32_t)*tp : 0u;
                tp += a.mn;
            }
        }
    }
    __device__ __forceinline__ uint32_t triple(const CrtTab& tab, int b, int i) const {
        if (PACK) return t[i];
        const int l = 12 * b + 3 * i, o = PACK ? 0 : 3 * i;
        return t[o] * tab.coef[l] + t[PACK ? 0 : o + 1] * tab.coef[l + 1] + t[PACK ? 0 : o + 2] * tab.coef[l + 2];
    }
};

// P_int of output e (two's complement, NW words)
template <int WG, int NW, bool PACK>
__device__ __forceinline__ void crt_sum(const CrtArgs& a, const CrtTab& tab, long long e, uint32_t (&X)[NW]) {
#pragma unroll
    for (int i = 0; i < NW; ++i) X[i] = 0;
    Fetch<PACK> cur;
    cur.load(a, tab, e, tab.G - 1, 0);
    for (int gi = tab.G - 1; gi >= 0; --gi) {
        uint64_t acc[WG];
#pragma unroll
        for (int k = 0; k < WG; ++k) acc[k] = 0;
        float F = 0.0f;
        // unrolled with a uniform exit: the table words are then immediate
        // constant operands of the products; the next four triples are in
        // flight while the last four are multiplied
        constexpr int NB = (MAXTRI + 3) / 4;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (4 * b >= tab.NT) break;
            Fetch<PACK> nxt;
            const bool more = b + 1 < NB && 4 * (b + 1) < tab.NT;
            if (more || gi > 0) nxt.load(a, tab, e, more ? gi : gi - 1, more ? b + 1 : 0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int q = 4 * b + i;
                if (q >= MAXTRI) break;
                const uint32_t u = cur.triple(tab, b, i);
#pragma unroll
                for (int k = 0; k < WG; ++k) acc[k] += (uint64_t)u * tab.Mt[q][k];
                F = fmaf((float)u, tab.inv[q], F);
            }
            cur = nxt;
        }
        // S_g = sum - R P (tab.Pneg = -P): the word sums as their low words plus
        // their high words one place up
        const uint32_t R = (uint32_t)rintf(F);
#pragma unroll
        for (int k = 0; k < WG; ++k) acc[k] += (uint64_t)R * tab.Pneg[k];
        uint32_t sg[WG];
        sg[0] = (uint32_t)acc[0];
        if (WG > 1) sg[WG > 1 ? 1 : 0] = add_first((uint32_t)acc[WG > 1 ? 1 : 0], (uint32_t)(acc[0] >> 32));
#pragma unroll
        for (int k = 2; k < WG; ++k) sg[k] = add_next((uint32_t)acc[k], (uint32_t)(acc[k - 1] >> 32));
        if (gi < tab.G - 1) shl_uniform<NW>(X, tab.w);
        const uint32_t sext = (uint32_t)((int)sg[WG - 1] >> 31);
        X[0] = add_first(X[0], sg[0]);
#pragma unroll
        for (int k = 1; k < NW; ++k) X[k] = add_next(X[k], k < WG ? sg[k < WG ? k : 0] : sext);
    }
}

// X += +-(x on the grid 2^E), Eq. (12): bits of x below the grid are dropped
template <int NW>
__device__ __forceinline__ void add_on_grid(uint32_t (&X)[NW], double x, int E, bool flip) {
    uint64_t mant;
    int e;
    bool neg;
    if (!decompose(x, mant, e, neg)) return;
    int s = e - 53 - E;
    if (s < 0) {
        mant = s <= -64 ? 0ull : mant >> -s;
        s = 0;
    }
    neg ^= flip;
    const int q = s >> 5, r = s & 31;
    const uint32_t f = neg ? 0xffffffffu : 0u;  // subtract as the complement plus one
    const uint32_t lo = (uint32_t)mant, hi = (uint32_t)(mant >> 32);
    const uint32_t p0 = (lo << r) ^ f, p1 = __funnelshift_l(lo, hi, r) ^ f, p2 = __funnelshift_l(hi, 0u, r) ^ f;
    add_first(f, f);  // the carry is set where neg
#pragma unroll
    for (int k = 0; k < NW; ++k)
        X[k] = add_next(X[k], k == q ? p0 : k == q + 1 ? p1 : k == q + 2 ? p2 : f);
}

// One output component: X holds n words below 2^(32 n), value (-1)^neg X
// 2^(top - 32 n), normalised here.  Writes RN to 53 bits, leaves the residual in
// the low n - 1 words with top and neg brought up to date.
template <int n, int NW>
__device__ __forceinline__ double next_component(uint32_t (&X)[NW], int& top, bool& neg) {
    // whole zero words (rare past the first component), then bits
    int moved = 0;
    while (X[n - 1] == 0u && moved < n) {
#pragma unroll
        for (int i = n - 1; i > 0; --i) X[i] = X[i - 1];
        X[0] = 0;
        ++moved;
    }
    if (X[n - 1] == 0u) return 0.0;  // nothing left
    const int z = __clz((int)X[n - 1]);
#pragma unroll
    for (int i = n - 1; i > 0; --i) X[i] = __funnelshift_l(X[i - 1], X[i], z);
    X[0] <<= z;
    top -= 32 * moved + z;
    const uint64_t v = ((uint64_t)X[n - 1] << 32) | X[n - 2];
    uint64_t q = v >> 11;
    uint32_t rest = X[n - 2] & 0x3ffu;
#pragma unroll
    for (int i = 0; i < n - 2; ++i) rest |= X[i];
    const bool up = (X[n - 2] & 0x400u) && (rest || (q & 1));
    X[n - 2] &= 0x7ffu;
    if (up) {
        q += 1;
        // the residual is 2^11 units of word n - 2 less the bits kept, of the opposite sign
        X[0] = add_first(~X[0], 1u);
#pragma unroll
        for (int i = 1; i < n - 1; ++i) X[i] = add_next(~X[i], 0u);
        X[n - 2] &= 0x7ffu;
    }
    // q 2^(top - 53), q in [2^52, 2^53]
    double x;
    if (top > -1021 && top < 1024) x = __longlong_as_double((long long)(((uint64_t)(top + 1021) << 52) + q));
    else x = scalbn((double)q, top - 53);
    // (the sign by its bit: a binary64 negation goes to the slow pipe)
    x = __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000u : 0), __double2loint(x));
    neg ^= up;
    top -= 32;  // word n - 2 is the new top word
    return x;
}

// The whole of one output; false (nothing written) when the old C needs more
// than NW words
template <int WG, int NW, bool PACK>
__device__ __forceinline__ bool crt_one(const CrtArgs& a, const CrtTab& tab, long long e) {
    int i, j;
    if (a.mn <= 0xffffffffll) {
        j = (int)((uint32_t)e / (uint32_t)a.m);
        i = (int)((uint32_t)e - (uint32_t)j * (uint32_t)a.m);
    } else {
        j = (int)(e / a.m);
        i = (int)(e - (long long)j * a.m);
    }
    double* cp = a.C + ((long long)i + (long long)j * a.ldc) * a.nc;
    int E = tab.w * tab.g0 - a.mu[i] - a.nu[j];
    double cl[4] = {0.0, 0.0, 0.0, 0.0};
    if (a.beta) {
        if (a.vec) {
            const double2 v = *(const double2*)cp;
            cl[0] = v.x;
            cl[1] = v.y;
            if (a.nc > 2) {
                const double2 u = *(const double2*)(cp + 2);
                cl[2] = u.x;
                cl[3] = u.y;
            }
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < a.nc) cl[c] = cp[c];
        }
    }
    const bool add = (__double_as_longlong(cl[0]) << 1) != 0;
    if (NW < WACC && add) {
        int eb = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) eb = max(eb, (__double2hiint(cl[c]) >> 20) & 0x7ff);
        if (eb - 1022 + 1 - E > 32 * NW - 2) return false;
    }
    uint32_t X[NW];
    crt_sum<WG, NW, PACK>(a, tab, e, X);
    const bool flip = a.alpha < 0;  // alpha X + C = alpha (X + alpha C)
    if (add) {
        if (NW == WACC) {
            // window: e_top = max(E0 + bitlen|P_int|, frexp_exp(C[0])) + 1; beyond
            // WINDOW_BITS the grid is raised and the product truncated toward zero
            const bool ng = (X[NW - 1] >> 31) != 0;
            negate_if<NW>(X, ng);
            const int etop = max(E + bit_length<NW>(X), frexp_exp(cl[0])) + 1;
            int d = etop - E - WINDOW_BITS;
            if (d > 0) {
                E += d;
                for (; d >= 32; d -= 32) {
#pragma unroll
                    for (int k = 0; k < NW - 1; ++k) X[k] = X[k + 1];
                    X[NW - 1] = 0;
                    if (d > 32 * NW) d = 32 * NW;
                }
#pragma unroll
                for (int k = 0; k < NW - 1; ++k) X[k] = __funnelshift_r(X[k], X[k + 1], d);
                X[NW - 1] >>= d;
            }
            negate_if<NW>(X, ng);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < a.nc) add_on_grid<NW>(X, cl[c], E, flip);
    }
    bool neg = (X[NW - 1] >> 31) != 0;
    negate_if<NW>(X, neg);
    neg ^= flip;
    int top = E + 32 * NW;
    cl[0] = next_component<NW, NW>(X, top, neg);
    cl[1] = next_component<NW - 1, NW>(X, top, neg);
    if (a.nc > 2) cl[2] = next_component<NW - 2, NW>(X, top, neg);
    if (a.nc > 3) cl[3] = next_component<NW - 3, NW>(X, top, neg);
    if (a.vec) {
        *(double2*)cp = make_double2(cl[0], cl[1]);
        if (a.nc > 2) *(double2*)(cp + 2) = make_double2(cl[2], cl[3]);
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < a.nc) cp[c] = cl[c];
    }
    return true;
}

template <int WG, bool PACK>
__device__ __noinline__ void crt_one_wide(const CrtArgs& a, const CrtTab& tab, long long e) {
    crt_one<WG, WACC, PACK>(a, tab, e);
}

template <int WG, int NW, bool PACK>
__global__ void __launch_bounds__(CT, min_blocks<NW, PACK>()) crt_kernel(const __grid_constant__ CrtArgs a,
                                                 const __grid_constant__ CrtTab tab) {
    chain_enter();
    const long long e = (long long)blockIdx.x * CT + threadIdx.x;
    if (e >= a.mn) return;
    if (!crt_one<WG, NW, PACK>(a, tab, e)) crt_one_wide<WG, PACK>(a, tab, e);
}

template <int WG, bool PACK>
void launch_crt_wg(const CrtArgs& a, const CrtTab& tab, cudaStream_t s) {
    const unsigned grid = (unsigned)((a.mn + CT - 1) / CT);
    // words for P_int with its sign and 30 bits or more above it for the old C
    const int need = (tab.pint_bits + 1 + 30 + 31) / 32;
#define OZLU_NW(W) \
    if (WG < W && need <= W) return launch(crt_kernel<WG, WG < W ? W : WACC, PACK>, grid, CT, 0, s, a, tab), void();
    OZLU_NW(10) OZLU_NW(11) OZLU_NW(12) OZLU_NW(13) OZLU_NW(14)
#undef OZLU_NW
    launch(crt_kernel<WG, WACC, PACK>, grid, CT, 0, s, a, tab);
}

template <bool PACK>
void launch_crt_pack(const CrtArgs& a, const CrtTab& tab, cudaStream_t s) {
    switch (tab.WG) {
#define OZLU_WG(W) case W: launch_crt_wg<W, PACK>(a, tab, s); break;
        OZLU_WG(5) OZLU_WG(6) OZLU_WG(7) OZLU_WG(8) OZLU_WG(9) OZLU_WG(10) OZLU_WG(11) OZLU_WG(12) OZLU_WG(13)
        OZLU_WG(14) OZLU_WG(15) OZLU_WG(16)
#undef OZLU_WG
        default: launch_crt_wg<4, PACK>(a, tab, s); break;
    }
}

}  // namespace
}  // namespace ozlu
