// (S1) shared exponents and (S2)+(S3) fused conversion of expansions to
// centered residue planes (Sec. 3.1, Sec. 3.2 Eq. (2), Sec. 3.3 Eq. (12)).
#include <limits.h>

#include "launch.cuh"
#include "conv_device.cuh"
#include "mp_device.cuh"
#include "ozlu_internal.h"

namespace ozlu {
namespace {

constexpr int NO_EXP = INT_MIN;

// (S1) of both operands in one launch.  Blocks [0, blocks_a): 32 rows of A each
// (consecutive rows are adjacent in memory, so a warp reads 32 of one column),
// 32 warps share the columns; the others: 32 columns of B each, one warp per
// column.  mu_i = (Q-1) - max_h frexp_exp(a_ih[0]), 0 for an all-zero row, nu_j
// likewise.  Bound by load latency: 32 warps a block and four loads in flight
// per thread (8 warps with one load each, one kernel a side, took 24 + 13 us at
// 3840 x 256).
// `clear` (may be null): the device error word, zeroed for a new call.
constexpr int SHIFT_THREADS = 1024;

__global__ void __launch_bounds__(SHIFT_THREADS) shift_kernel(const double* A, long long lda, int m,
                                                              const double* B, long long ldb, int n,
                                                              int nc, int k, int Q, int* mu,
                                                              int* nu, int blocks_a, int* clear) {
    chain_enter();
    __shared__ int red[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0;
    int E = NO_EXP;
    if ((int)blockIdx.x < blocks_a) {
        const int i = blockIdx.x * 32 + lane;
        if (i < m) {
            const double* x = A + (long long)i * nc;
            const long long step = lda * nc;
#pragma unroll 4
            for (int h = warp; h < k; h += 32) {
                const double v = *(x + h * step);
                if (v != 0.0) E = max(E, frexp_exp(v));
            }
        }
        red[warp][lane] = E;
        __syncthreads();
        if (warp == 0 && i < m) {
#pragma unroll
            for (int r = 1; r < 32; ++r) E = max(E, red[r][lane]);
            mu[i] = E == NO_EXP ? 0 : (Q - 1) - E;
        }
    } else {
        const int j = ((int)blockIdx.x - blocks_a) * 32 + warp;
        if (j >= n) return;
        const double* x = B + (long long)j * ldb * nc;
#pragma unroll 4
        for (int h = lane; h < k; h += 32) {
            const double v = *(x + (long long)h * nc);
            if (v != 0.0) E = max(E, frexp_exp(v));
        }
        E = __reduce_max_sync(0xffffffffu, E);
        if (lane == 0) nu[j] = E == NO_EXP ? 0 : (Q - 1) - E;
    }
}

constexpr int MAXD = 9;  // words of one balanced digit (w + 2 bits)

// Residue modulo a binary64-back-end prime (m < 2^27): 64-bit sum of the
// half products, then one 64-bit remainder.
template <int H>
__device__ __forceinline__ int centered_residue64(const uint32_t (&mag)[MAXD], bool neg,
                                                  const DevTable& tab, int l) {
    const uint64_t m = (uint64_t)tab.mod[l];
    uint64_t acc = 0;
#pragma unroll
    for (int j = 0; j < H; ++j) {
        const uint64_t half = (mag[j >> 1] >> (16 * (j & 1))) & 0xffffu;
        acc += half * tab.pow16[l][j];
    }
    uint64_t r = acc % m;
    if (neg && r) r = m - r;
    long long c = (long long)r;
    if (c > (long long)(m - 1) / 2) c -= (long long)m;
    return (int)c;
}

// Binary64 back-end.  One element per thread: x -> X = Eq. (12) -> S balanced
// digits (Eq. (2)) -> centered residues for every modulus, as doubles.
//   A side (is_b = 0): element (r, h) of an R x K matrix, plane [l][t][r][h]
//   B side (is_b = 1): element (h, r) of a K x R matrix, plane [l][t][r][h]
// Threads cover [0, R) x [0, Kpad) and write zeros in the K padding; the
// padded rows are left as they are (they only reach discarded outputs).
template <int H>
__global__ void __launch_bounds__(256) convert64_kernel(
    const double* X, long long ld, int nc, int R, int K, int is_b,
    const int* shifts, const __grid_constant__ DevTable tab, int Kpad, int Rpad,
    double* planes) {
    chain_enter();
    const int h = blockIdx.x * 32 + (threadIdx.x & 31);
    const int r = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (h >= Kpad || r >= R) return;
    const size_t plane = (size_t)Rpad * Kpad;
    const size_t off = (size_t)r * Kpad + h;
    if (h >= K) {
        for (int l = 0; l < tab.N; ++l)
            for (int t = 0; t < tab.S; ++t) planes[(size_t)(l * tab.S + t) * plane + off] = 0.0;
        return;
    }
    const double* x = is_b ? X + ((long long)h + (long long)r * ld) * nc
                           : X + ((long long)r + (long long)h * ld) * nc;
    const int shift = shifts[r];
    uint32_t V[MAXWX];
#pragma unroll
    for (int wd = 0; wd < MAXWX; ++wd) V[wd] = 0;
    for (int c = 0; c < nc; ++c) add_component<MAXWX>(V, x[c], shift);

    const int w = tab.w, S = tab.S;
    const int nw = (w + 2 + 31) >> 5;  // words of a digit with its carry
    uint32_t carry = 0;
    for (int t = 0; t < S; ++t) {
        uint32_t D[MAXD];
#pragma unroll
        for (int k2 = 0; k2 < MAXD; ++k2) D[k2] = 0;
        bool neg = false;
        if (t < S - 1) {
            // unsigned field [t w, t w + w) plus the incoming carry
#pragma unroll
            for (int k2 = 0; k2 < MAXD; ++k2)
                if (k2 < nw) D[k2] = field32<MAXWX>(V, t * w + 32 * k2);
            mask_below<MAXD>(D, w);
            uint64_t c = carry;
#pragma unroll
            for (int k2 = 0; k2 < MAXD; ++k2) {
                const uint64_t s = (uint64_t)D[k2] + c;
                D[k2] = (uint32_t)s;
                c = s >> 32;
            }
            // balanced: D >= 2^(w-1) -> digit D - 2^w (negative), carry out 1
            const bool big = bit_at<MAXD>(D, w - 1) || bit_at<MAXD>(D, w);
            if (big) {
                complement_below<MAXD>(D, w);  // |digit| = 2^w - D (0 when D = 2^w)
                neg = true;
                carry = 1;
            } else {
                carry = 0;
            }
            // D = 2^w exactly (field all ones plus carry) gives digit 0
        } else {
            // top digit: signed field from bit t w upward, plus the carry
            uint32_t T[MAXD + 1];
#pragma unroll
            for (int k2 = 0; k2 <= MAXD; ++k2) T[k2] = field32<MAXWX>(V, t * w + 32 * k2);
            uint64_t c = carry;
#pragma unroll
            for (int k2 = 0; k2 <= MAXD; ++k2) {
                const uint64_t s = (uint64_t)T[k2] + c;
                T[k2] = (uint32_t)s;
                c = s >> 32;
            }
            neg = (T[MAXD] >> 31) != 0;
            if (neg) negate<MAXD + 1>(T);
#pragma unroll
            for (int k2 = 0; k2 < MAXD; ++k2) D[k2] = T[k2];
        }
        for (int l = 0; l < tab.N; ++l)
            planes[(size_t)(l * S + t) * plane + off] = (double)centered_residue64<H>(D, neg, tab, l);
    }
}

// ---------------------------------------------------------------------------
// (S2)+(S3) for moduli <= 255, both operands in one launch.  A thread takes E
// consecutive positions h of one plane row r (A side: elements (r, h) of A,
// B side: elements (h, r) of B), forms X (Eq. (12)) in NWX words, and takes
// one digit at a time off its low end (Eq. (2)).  Bound by integer issue: a
// residue is NW four-byte dot products against the bytes 2^(8 j) mod m, one
// exact high-word reduction and the packing, about 9 instructions, where the
// former kernel (16-bit halves, one element a thread, sign fixed up after the
// reduction) took about 30.  The table words of a modulus are uniform over the
// warp and are read once for E elements; E results are stored as one word.
// Exponents and conversion of both operands, QD, 3840 x 256 each to FP16: 162 us
// (343 before); 1024 x 1024 to FP8: 224 us (449 before).
//   E = 4 where that still leaves two blocks of 256 threads per SM, else E = 1
//   and the moduli split over gridDim.y (X formed again in each slice).
// Positions h >= K (the K padding) come out as zeros; the rows beyond R are
// left as they are (they only reach discarded outputs).
template <int NWX>
__device__ __forceinline__ void shift_down(uint32_t (&V)[NWX], int w) {
    const uint32_t sext = (uint32_t)((int)V[NWX - 1] >> 31);
    const int q = w >> 5;
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1)
        if (s < NWX && (q & s)) {
#pragma unroll
            for (int i = 0; i < NWX; ++i) V[i] = i + s < NWX ? V[i + s < NWX ? i + s : 0] : sext;
        }
#pragma unroll
    for (int i = 0; i < NWX; ++i) V[i] = __funnelshift_r(V[i], i + 1 < NWX ? V[i + 1 < NWX ? i + 1 : 0] : sext, w & 31);
}

struct ConvArgs {
    const double* A;
    const double* B;
    long long lda, ldb;
    const int* mu;
    const int* nu;
    void* RA;
    void* RB;
    int m, n, K, nc, Kpad, Mpad, Npad;
    int blocks_a;  // blocks of the A side; the B side follows
    int lper;      // moduli per gridDim.y slice
};

template <int MODE, int NWX, int NW, int E>
__global__ void __launch_bounds__(256) convert_kernel(const __grid_constant__ ConvArgs a,
                                                      const __grid_constant__ ConvTab tab) {
    chain_enter();
    const bool is_b = (int)blockIdx.x >= a.blocks_a;
    const int HG = a.Kpad / E;
    const long long idx = (long long)((int)blockIdx.x - (is_b ? a.blocks_a : 0)) * 256 + threadIdx.x;
    const int r = (int)(idx / HG), h0 = (int)(idx - (long long)r * HG) * E;
    if (r >= (is_b ? a.n : a.m)) return;
    const size_t plane = (size_t)(is_b ? a.Npad : a.Mpad) * a.Kpad;
    const size_t off = (size_t)r * a.Kpad + h0;
    uint32_t V[E][NWX];
    {
        const int shift = is_b ? a.nu[r] : a.mu[r];
        const long long step = is_b ? a.nc : a.lda * a.nc;
        const double* x = is_b ? a.B + (h0 + (long long)r * a.ldb) * a.nc : a.A + (r + (long long)h0 * a.lda) * a.nc;
#pragma unroll
        for (int e = 0; e < E; ++e) {
#pragma unroll
            for (int i = 0; i < NWX; ++i) V[e][i] = 0;
            if (h0 + e < a.K)
                for (int c = 0; c < a.nc; ++c) add_component<NWX>(V[e], *(x + e * step + c), shift);
        }
    }
    const int S = tab.S, w = tab.w;
    const int l0 = blockIdx.y * a.lper, l1 = min(tab.N, l0 + a.lper);
    const uint32_t mk = (1u << (w - 32 * (NW - 1))) - 1u;  // bits of the digit's last word below w
    uint32_t carry[E];
#pragma unroll
    for (int e = 0; e < E; ++e) carry[e] = 0;
    for (int t = 0; t < S; ++t) {
        const bool top = t == S - 1;
        uint32_t D[E][NW], wf[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            wf[e] = top ? V[e][NWX - 1] >> 31 : 0u;
            uint64_t c = carry[e];
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                uint32_t v = V[e][i < NWX ? i : NWX - 1];
                if (!top && i == NW - 1) v &= mk;
                c += v;
                D[e][i] = (uint32_t)c;
                c >>= 32;
            }
            if (top) {
                // two's complement over NW words; -1 plus the carry is 0
                if (c) wf[e] = 0;
            } else {
                // balanced: D >= 2^(w-1) stands for D - 2^w and carries one
                uint32_t hi = 0;
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    if (i == ((w - 1) >> 5)) hi |= D[e][i] >> ((w - 1) & 31);
                    if (i == (w >> 5)) hi |= D[e][i] >> (w & 31);
                }
                wf[e] = hi & 1u;
                carry[e] = wf[e];
                shift_down<NWX>(V[e], w);
            }
        }
        for (int l = l0; l < l1; ++l) {
            const ConvMod& M = tab.mod[l];
            const uint32_t wc = top ? M.topc : M.wrapc;
            uint32_t res[E];  // centered residue + half
#pragma unroll
            for (int e = 0; e < E; ++e) res[e] = conv_residue<NW>(D[e], M, wf[e] * wc + M.half);
            store_residues<MODE, E>(is_b ? a.RB : a.RA, (size_t)(l * S + t), plane, off, M, res);
        }
    }
}

template <int MODE, int NWX, int NW>
void launch_conv(ConvArgs a, const ConvTab& t, cudaStream_t s) {
    const long long work = ((long long)a.m + a.n) * a.Kpad;
    const int sms = device_sms();
    if (NWX <= 8 && work >= 4ll * 512 * sms) {
        constexpr int E = NWX <= 8 ? 4 : 1;
        const long long ta = (long long)a.m * (a.Kpad / E), tb = (long long)a.n * (a.Kpad / E);
        a.blocks_a = (int)((ta + 255) / 256);
        a.lper = t.N;
        launch(convert_kernel<MODE, NWX, NW, E>, a.blocks_a + (unsigned)((tb + 255) / 256), 256, 0, s, a, t);
        return;
    }
    const long long ta = (long long)a.m * a.Kpad, tb = (long long)a.n * a.Kpad;
    a.blocks_a = (int)((ta + 255) / 256);
    const int blocks = a.blocks_a + (int)((tb + 255) / 256);
    // few elements: the moduli over up to 8 slices, X and its digits formed in each
    int split = (2 * sms + blocks - 1) / blocks;
    if (split > 8) split = 8;
    if (split > t.N) split = t.N;
    a.lper = (t.N + split - 1) / split;
    launch(convert_kernel<MODE, NWX, NW, 1>, dim3(blocks, (t.N + a.lper - 1) / a.lper), 256, 0, s, a, t);
}

template <int MODE>
void launch_conv_mode(const ConvArgs& a, const ConvTab& t, cudaStream_t s) {
    // X in 8 words covers every expansion up to 255 bits (QD with its slack);
    // wider ones (large guard settings) take 12
    switch ((t.WX > 8 ? 16 : 0) + t.NW) {
#define OZLU_CONV(NN)                                                   \
    case NN: launch_conv<MODE, 8, NN>(a, t, s); break;                  \
    case 16 + NN: launch_conv<MODE, 12, NN>(a, t, s); break;
        OZLU_CONV(1) OZLU_CONV(2) OZLU_CONV(3) OZLU_CONV(4) OZLU_CONV(5) OZLU_CONV(6) OZLU_CONV(7) OZLU_CONV(8)
#undef OZLU_CONV
    }
}

}  // namespace

void launch_shifts(const double* A, long long lda, int m, const double* B, long long ldb, int n, int nc, int k, int Q,
                   int* mu, int* nu, int* clear, cudaStream_t s) {
    const int ba = (m + 31) / 32, bb = (n + 31) / 32;
    launch(shift_kernel, ba + bb, SHIFT_THREADS, 0, s, A, lda, m, B, ldb, n, nc, k, Q, mu, nu, ba, clear);
}

void launch_convert(const double* A, long long lda, int m, const double* B, long long ldb, int n, int nc, int k,
                    const int* mu, const int* nu, const ConvTab& t, int Kpad, int Mpad, int Npad, void* RA, void* RB,
                    int mode, cudaStream_t s) {
    const ConvArgs a{A, B, lda, ldb, mu, nu, RA, RB, m, n, k, nc, Kpad, Mpad, Npad, 0, 0};
    if (mode == 0) launch_conv_mode<0>(a, t, s);
    else if (mode == 1) launch_conv_mode<1>(a, t, s);
    else launch_conv_mode<2>(a, t, s);
}

void launch_convert64(const double* X, long long ld, int nc, int rows, int cols, bool is_b, const int* shifts,
                      const DevTable& tab, int Kpad, int Rpad, double* planes, cudaStream_t s) {
    // A side: rows = R, cols = K; B side: rows = K, cols = R
    const int R = is_b ? cols : rows;
    const int K = is_b ? rows : cols;
    // rows [0, R) only: padded rows only feed padded output rows and columns,
    // which the epilogue discards; the padded K columns must be zero
    dim3 grid((Kpad + 31) / 32, (R + 7) / 8);
    if (R == 0) return;
    switch (tab.H) {
#define OZLU_CONV(HH) \
    case HH: \
        launch(convert64_kernel<HH>, grid, 256, 0, s, X, ld, nc, R, K, is_b ? 1 : 0, shifts, tab, Kpad, Rpad, planes); \
        break;
        OZLU_CONV(2) OZLU_CONV(3) OZLU_CONV(4) OZLU_CONV(5) OZLU_CONV(6)
        OZLU_CONV(7) OZLU_CONV(8) OZLU_CONV(9) OZLU_CONV(10) OZLU_CONV(11) OZLU_CONV(12)
        OZLU_CONV(13) OZLU_CONV(14) OZLU_CONV(15)
#undef OZLU_CONV
        default:
            launch(convert64_kernel<16>, grid, 256, 0, s, X, ld, nc, R, K, is_b ? 1 : 0, shifts, tab, Kpad, Rpad, planes);
    }
}

}  // namespace ozlu
