// The cooperative panel kernel of the LU (lu.cu), with its exchange of tagged words.
#pragma once

#include <stdint.h>

#include "../../include/ozlu.h"
#include "mpf.cuh"

namespace ozlu {
namespace {

constexpr int PBASE = 128;      // widest base block of the cooperative panel kernel

// limbs of the panel arithmetic: 32 L >= 53 nc + 12 (DD 4, TD 6, QD 7)
template <int N>
struct Limbs { static constexpr int L = N == 2 ? 4 : (N == 3 ? 6 : 7); };

__device__ __forceinline__ double* elem(double* A, long long lda, int nc, long long i, long long j) {
    return A + (i + j * lda) * nc;
}

// Cooperative factorisation of one base block: columns [c0, c0 + b) over rows
// [c0, n).  One block per SM owns a contiguous slice of rows and keeps its
// b-column slice in shared memory as L-limb floats for the whole block.
//
// A column is a serial chain (the pivot, its reciprocal, the next column, the
// next candidate) through every block, so the kernel is bound by latency, and
// what is off the chain runs beside it on warps of its own:
//   warp 0      the chain: reduce the blocks' keys to the pivot, fetch the
//               pivot's reciprocal and its next element, update the next column,
//               choose and announce the block's candidate, invert it;
//   warp 1      the multipliers; then column kc + 2, which the chain needs next;
//   warps 2, 3  the pivot row into shared memory, the interchange;
//   warps 4 ..  the trailing update of the last column, then the two rows other
//               blocks may need from this one (its candidate and the row the
//               pivot will replace), published as they are formed.
// The next column is updated as y - l u with the multiplier l = x (1 / p) that is
// stored, one rounding like every other element; l is formed again on warp 0 when
// the reciprocal arrives.  (y - (x u) (1 / p), with x u ready by then, is a product
// shorter on the chain, QD n = 1000 / 4096 6.63 / 50.7 ms against 6.68 / 50.9, but
// rounds both factors: backward error of the n = 4096 LU at cond 1e40, sampled,
// 1.74e-66 against 1.39e-66.)
//
// Blocks exchange 64-bit words whose upper half is a tag (the column) and whose
// lower half is data, so that a word announces itself: readers poll the words
// they need, and neither side pays for a fence (about 1000 cycles each at GPU
// scope).  Only relaxed accesses to single words are used.  The first word a
// block announces is its candidate's key, before its row is final.  There are
// three slots per block, used in turn: a block writes the words of column kc + 3
// only after every block has announced its key of kc + 2, which a block does after
// the block-wide barrier of column kc, i.e. when all its warps have read what they
// need of column kc.  The words are zeroed before every factorisation and tags are
// column numbers, so a stale word never matches.
//
// Measured, QD panels of the n = 1000 / 4096 LU (nb = 256): 4.2 / 21.6 ms (4.2 us a
// column at n = 1000), from 13.0 / 58.7 ms with a stamp over a fenced row and the
// exchange, the reciprocal and the multipliers on the same warp in turn.
//
// The interchanges of the columns outside the base block are applied once,
// after the last column, as one permutation (laswp2; by one thread per column
// swap by swap they took 150 us per 128 columns).  Every wait is bounded (2 s of
// the global timer); on expiry the kernel records OZLU_ERR_TIMEOUT in the
// scratch and every block returns.
constexpr int COOP_MAXG = 304;           // blocks (up to 2 per SM)
constexpr int COOP_THREADS = 512;
constexpr int COOP_DEPTH = 3;            // slots per block
constexpr unsigned long long COOP_WAIT_NS = 2000000000ull;

// stamp word of a slot: bits 63..44 the column (c0 + kc + 1, modulo 2^20),
// bits 43..0 the candidate's key (mpf_key; 0: no candidate)
constexpr int STAMP_SHIFT = 44;
constexpr unsigned long long KEY_MASK = (1ull << STAMP_SHIFT) - 1;

// tagged words: (tag << 32) | data, tag = c0 + kc + 1
template <int L>
struct CoopSlot {
    static constexpr int WORDS = L + 2;       // MPF: limbs, exponent, sign
    unsigned long long stamp;
    unsigned long long idx;                   // the candidate's global row
    unsigned long long rec[WORDS];            // 1 / the candidate (0 for a zero candidate)
    unsigned long long row[WORDS][PBASE];     // the candidate row (all b columns), word-major
};

template <int L>
struct CoopScratch {
    int error;
    int pad[3];
    CoopSlot<L> part[COOP_DEPTH][COOP_MAXG];             // by column modulo COOP_DEPTH
    unsigned long long orow[COOP_DEPTH][L + 2][PBASE];   // old row c, for the owner of the pivot row
};

#if defined(__CUDACC__)
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// named barriers of the kernel below: the count of threads that arrive or wait
// (whole warps, converged)
__device__ __forceinline__ void bar_sync(int id, int threads) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
#endif  // (a CPU build of the kernel, for tests, brings its own)

// The bound of a wait, for a polling loop that calls expired() once per failed
// poll: true after limit_ns of the global timer (the error word is then set) or
// when another block has given up.  The timer, slow to read, is first read
// after 256 polls.
struct WaitBound {
    unsigned long long t0 = 0;
    int it = 0;
    __device__ __forceinline__ bool expired(int* err, unsigned long long limit_ns = COOP_WAIT_NS) {
        if ((++it & 255) != 0) return false;
        if (*(volatile int*)err) return true;
        const unsigned long long t = global_ns();
        if (it == 256) t0 = t;
        if (t - t0 <= limit_ns) return false;
        atomicExch(err, OZLU_ERR_TIMEOUT);
        return true;
    }
};

// wait until the stamp word carries column `want`; returns it, or 0 on expiry
__device__ __forceinline__ unsigned long long wait_stamp(const unsigned long long* p, unsigned want,
                                                         int* err,
                                                         unsigned long long limit_ns = COOP_WAIT_NS) {
    WaitBound wb;
    for (;;) {
        const unsigned long long v = ld_relaxed(p);
        if ((unsigned)(v >> STAMP_SHIFT) == want) return v;
        if (wb.expired(err, limit_ns)) return 0;
    }
}

// Poll n tagged words a lane (p[i], skipped where null) until all carry `tag`;
// false on expiry.  All loads of a round are in flight together.  The lanes
// decide together, so a warp leaves the loop converged.
template <int n>
__device__ __forceinline__ bool wait_words(const unsigned long long* const (&p)[n], unsigned tag, uint32_t (&v)[n],
                                           int* err) {
    WaitBound wb;
    unsigned long long w[n];
#pragma unroll
    for (int i = 0; i < n; ++i) w[i] = 0;
    for (;;) {
        bool miss = false;
#pragma unroll
        for (int i = 0; i < n; ++i)
            if (p[i] && (unsigned)(w[i] >> 32) != tag) w[i] = ld_relaxed(p[i]);
#pragma unroll
        for (int i = 0; i < n; ++i) {
            v[i] = (uint32_t)w[i];
            miss |= p[i] && (unsigned)(w[i] >> 32) != tag;
        }
        if (!__any_sync(0xffffffffu, miss)) return true;
        if (__any_sync(0xffffffffu, wb.expired(err))) return false;
    }
}

// word i of an L-limb float (limbs, exponent, sign) and its inverse
template <int L>
__device__ __forceinline__ uint32_t mpf_word(const MPF<L>& v, int i) {
    return i < L ? v.m[i < L ? i : 0] : (uint32_t)(i == L ? v.e : v.neg);
}

// the float whose word i lane i holds, on every lane
template <int L>
__device__ __forceinline__ MPF<L> mpf_gather(uint32_t w) {
    MPF<L> v;
#pragma unroll
    for (int i = 0; i < L; ++i) v.m[i] = __shfl_sync(0xffffffffu, w, i);
    v.e = (int)__shfl_sync(0xffffffffu, w, L);
    v.neg = (int)__shfl_sync(0xffffffffu, w, L + 1);
    return v;
}

// x = v where `on`, by selects
template <int L>
__device__ __forceinline__ void mpf_take(MPF<L>& x, const MPF<L>& v, bool on) {
#pragma unroll
    for (int i = 0; i < L; ++i) x.m[i] = on ? v.m[i] : x.m[i];
    x.e = on ? v.e : x.e;
    x.neg = on ? v.neg : x.neg;
}

// lane src's float on every lane
template <int L>
__device__ __forceinline__ MPF<L> mpf_bcast(const MPF<L>& x, int src) {
    MPF<L> v;
#pragma unroll
    for (int i = 0; i < L; ++i) v.m[i] = __shfl_sync(0xffffffffu, x.m[i], src);
    v.e = __shfl_sync(0xffffffffu, x.e, src);
    v.neg = __shfl_sync(0xffffffffu, x.neg, src);
    return v;
}

// 44-bit order key of |v|: exponent (12 bits), then the top limb (values are
// normalised); a larger key means a larger |v|, equal keys need the full
// comparison.  An exact zero gets 1 (below every nonzero value, above "no
// candidate" = 0).  Exponents outside [-2047, 2047] share the lowest or the
// highest nonzero key, so that they always go through the full comparison.
template <int L>
__device__ __forceinline__ unsigned long long mpf_key(const MPF<L>& v) {
    // (selects, so that the lanes of a warp stay together)
    const unsigned hi = v.e < -2047 ? 1u : (v.e > 2047 ? 0xfffu : (unsigned)(v.e + 2048));
    const unsigned lo = v.e < -2047 ? 0u : (v.e > 2047 ? 0xffffffffu : v.m[L - 1]);
    const unsigned long long k = ((unsigned long long)hi << 32) | lo;
    return mpf_zero<L>(v) ? 1ull : k;
}

// |a| > |b|, or equal and ia < ib (first index on ties); ib < 0: b is empty
template <int L>
__device__ __forceinline__ bool mpf_better(const MPF<L>& a, int ia, const MPF<L>& b, int ib) {
    if (ia < 0) return false;
    if (ib < 0) return true;
    const int c = mpf_abs_cmp<L>(a, b);
    return c > 0 || (c == 0 && ia < ib);
}

// warp-wide argmax of (|v|, first index): every lane ends with the winner
template <int L>
__device__ __forceinline__ void warp_best(MPF<L>& v, int& idx, int& aux) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        MPF<L> w;
#pragma unroll
        for (int q = 0; q < L; ++q) w.m[q] = __shfl_xor_sync(0xffffffffu, v.m[q], o);
        w.e = __shfl_xor_sync(0xffffffffu, v.e, o);
        w.neg = __shfl_xor_sync(0xffffffffu, v.neg, o);
        const int wi = __shfl_xor_sync(0xffffffffu, idx, o);
        const int wa = __shfl_xor_sync(0xffffffffu, aux, o);
        if (mpf_better<L>(w, wi, v, idx)) { v = w; idx = wi; aux = wa; }
    }
}

// warp-wide max of (key, then lowest index >= 0) by three integer reductions;
// idx < 0: none (its key is 0)
__device__ __forceinline__ void warp_best_key(unsigned long long& k, int& idx) {
    const unsigned hi = idx >= 0 ? (unsigned)(k >> 32) : 0u;
    const unsigned H = __reduce_max_sync(0xffffffffu, hi);
    const unsigned lo = idx >= 0 && hi == H ? (unsigned)k : 0u;
    const unsigned Lo = __reduce_max_sync(0xffffffffu, lo);
    const bool mine = idx >= 0 && hi == H && (unsigned)k == Lo;
    idx = (int)__reduce_min_sync(0xffffffffu, mine ? (unsigned)idx : 0xffffffffu);
    k = ((unsigned long long)H << 32) | Lo;
}

// Q: rows of warp 0's lanes, nr <= 32 Q
template <int N, int Q>
__global__ void __launch_bounds__(COOP_THREADS, 1) base_block_coop_kernel(
    double* A, long long lda, int n, int c0, int b, int rows_per_block, int* ipiv, int* info,
    CoopScratch<Limbs<N>::L>* sc) {
    constexpr int L = Limbs<N>::L, WORDS = L + 2;
    constexpr int T = COOP_THREADS;
    constexpr int BAR_PIVOT = 1;  // warps 0 .. 3: the pivot's slot is known
    constexpr int BAR_COL = 2;    // column kc + 2 is updated (warp 0 waits, the others arrive)
    constexpr int BAR_ROWS = 3;   // the pair of rows is published (warps 1 .. 3 wait, its publishers arrive)
    constexpr int ROWS_T = (3 + 8) * 32;
    extern __shared__ __align__(16) unsigned char smraw[];
    MPF<L>* a = reinterpret_cast<MPF<L>*>(smraw);  // [r][k], r < rows_per_block, k < b
    // rows padded to b + 1 entries: threads on consecutive rows of one column
    // then fall on different shared-memory banks
    const int bs = b + 1;
    __shared__ MPF<L> prow[2][PBASE];  // the pivot row, double-buffered by column parity
    __shared__ int s_cand, s_slot, s_zero;
    __shared__ int s_fail[2];  // by column parity: a slow warp still reads the last one
    const int g = blockIdx.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31;
    // (broadcast, so that the compiler sees the warps' branches as uniform: it
    // then keeps shuffles and reductions in them inline; else each takes an
    // out-of-line reconvergence, about 250 cycles)
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int r0 = c0 + g * rows_per_block;
    const int r1 = min(n, r0 + rows_per_block);
    const int nr = max(0, r1 - r0);
    auto owns = [&](int row) { return row >= r0 && row < r1; };
    int* err = &sc->error;

    if (tid < 2) s_fail[tid] = 0;
    for (int p = tid; p < nr * b; p += T) {
        const int r = p / b, k = p - r * b;
        a[r * bs + k] = mpf_from_exp<L, N>(elem(A, lda, N, r0 + r, c0 + k));
    }
    __syncthreads();

    // warp 0: the block's candidate among the rows >= row_lo for column kc, whose
    // values the lanes hold (v[q]: row lane + 32 q); announces it and leaves its
    // row in s_cand; returns its value
    auto choose = [&](const MPF<L> (&v)[Q], int row_lo, int kc) -> MPF<L> {
        unsigned long long bk = 0;
        int bi = -1;
        MPF<L> mine = v[0];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (32 * q >= nr) break;
            const int r = lane + 32 * q;
            const bool in = r < nr && r0 + r >= row_lo;
            const unsigned long long k = mpf_key<L>(v[q]);
            bool better = in && (bi < 0 || k > bk);
            if (q > 0 && __any_sync(0xffffffffu, in && bi >= 0 && k == bk))
                better = better || (in && bi >= 0 && k == bk && mpf_abs_cmp<L>(v[q], mine) > 0);
            bk = better ? k : bk;
            bi = better ? r0 + r : bi;
            if (q > 0) {
#pragma unroll
                for (int i = 0; i < L; ++i) mine.m[i] = better ? v[q].m[i] : mine.m[i];
                mine.e = better ? v[q].e : mine.e;
                mine.neg = better ? v[q].neg : mine.neg;
            }
        }
        __syncwarp();
        unsigned long long K = bk;
        int I = bi;
        warp_best_key(K, I);
        if (__any_sync(0xffffffffu, bi >= 0 && bk == K && bi != I)) {  // equal keys: compare exactly
            MPF<L> x = (bi >= 0 && bk == K) ? mine : mpf_make_zero<L>();
            int xi = (bi >= 0 && bk == K) ? bi : -1, aux = 0;
            warp_best<L>(x, xi, aux);
            I = xi;
        }
        const unsigned tag = (unsigned)(c0 + kc + 1);
        CoopSlot<L>& slot = sc->part[kc % COOP_DEPTH][g];
        if (lane == 0) {
            st_relaxed(&slot.stamp, ((unsigned long long)(tag & 0xfffff) << STAMP_SHIFT) | (I >= 0 ? K : 0ull));
            st_relaxed(&slot.idx, ((unsigned long long)tag << 32) | (unsigned)I);
            s_cand = I;
        }
        const MPF<L> best = mpf_bcast<L>(mine, I >= 0 ? (I - r0) & 31 : 0);
        return I >= 0 ? best : mpf_make_zero<L>();
    };
    // warp 0: the reciprocal of the candidate of column kc
    auto publish_rec = [&](const MPF<L>& cand, int kc) {
        const MPF<L> r = mpf_zero<L>(cand) ? mpf_make_zero<L>() : mpf_recip<L>(cand);
        uint32_t w = 0;
#pragma unroll
        for (int i = 0; i < WORDS; ++i) w = lane == i ? mpf_word<L>(r, i) : w;
        if (lane < WORDS)
            st_relaxed(&sc->part[kc % COOP_DEPTH][g].rec[lane], ((unsigned long long)(unsigned)(c0 + kc + 1) << 32) | w);
    };
    // four warps each for the candidate row (pub 0 .. 3) and, in its owner, row
    // c0 + kc + 1 (pub 4 .. 7): update it by column kc (kc < 0 or zero: no update)
    // and publish it for column kc + 1.  None of them shares warp 0's scheduler,
    // where the reciprocal runs at the same time.  They read and write the two rows
    // in shared memory, which the next column's multipliers and interchange write
    // too: those wait for them at BAR_ROWS (a word in the exchange says that its own
    // element is done, not that the row's multiplier has been read by all).
    const int pub = (warp & 3) == 0 || warp < 5 || warp > 14 ? -1 : (warp - 5) - ((warp - 5) >> 2);
    auto publish_rows = [&](int kc, bool zero, int pa, int pb) {
        const unsigned long long tag = (unsigned long long)(unsigned)(c0 + kc + 2) << 32;
        const int r = pub < 4 ? pa : pb, k = (pub & 3) * 32 + lane;
        if (r < 0 || (pub >= 4 && pb == pa)) return;
        unsigned long long* orow = &sc->orow[(kc + 1) % COOP_DEPTH][0][0];
        unsigned long long* dst = pub < 4 ? &sc->part[(kc + 1) % COOP_DEPTH][g].row[0][0] : orow;
        if (k < b) {
            MPF<L> v = a[r * bs + k];
            if (!zero && k >= kc + 2) {
                v = mpf_fms_oolv<L>(v, a[r * bs + kc], prow[kc & 1][k]);
                a[r * bs + k] = v;
            }
#pragma unroll
            for (int i = 0; i < WORDS; ++i) st_relaxed(dst + i * PBASE + k, tag | mpf_word<L>(v, i));
            if (pb == pa) {  // the candidate is row c0 + kc + 1 itself
#pragma unroll
                for (int i = 0; i < WORDS; ++i) st_relaxed(orow + i * PBASE + k, tag | mpf_word<L>(v, i));
            }
        }
    };

    MPF<L> cand = mpf_make_zero<L>();  // warp 0: this block's candidate
    if (warp == 0) {
        MPF<L> v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = lane + 32 * q < nr ? a[(lane + 32 * q) * bs] : mpf_make_zero<L>();
        cand = choose(v, c0, 0);
    }
    __syncthreads();
    if (warp == 0) {
        publish_rec(cand, 0);
    } else {
        if (pub >= 0) {
            publish_rows(-1, true, s_cand >= 0 ? s_cand - r0 : -1, owns(c0) ? c0 - r0 : -1);
            bar_arrive(BAR_ROWS, ROWS_T);
        }
        bar_arrive(BAR_COL, T);
    }

    // the trailing update by column bulk_kc of the rows outside the pair that
    // publish_rows took is deferred to the next column (bulk_kc < 0: none)
    int bulk_kc = -1, bulk_lo = 0, bulk_pa = -1, bulk_pb = -1;
    for (int kc = 0; kc < b; ++kc) {
        const int c = c0 + kc;
        const unsigned tag = (unsigned)(c + 1);
        MPF<L>* pr = prow[kc & 1];
        const int lo = max(r0, c + 1) - r0;  // first row below the pivot
        const bool last = kc == b - 1;
        const unsigned long long* orow = &sc->orow[kc % COOP_DEPTH][0][0];
        if (warp == 0) {
            // the rows' elements of column kc, before warp 1 makes them multipliers
            MPF<L> x[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (lane + 32 * q < nr) x[q] = a[(lane + 32 * q) * bs + kc];
                else x[q] = mpf_make_zero<L>();
            // every block's key of column kc
            constexpr int PER = (COOP_MAXG + 31) / 32;
            const unsigned want = tag & 0xfffff;
            unsigned long long key[PER];
            WaitBound wb;
            bool ok = true;
#pragma unroll
            for (int u = 0; u < PER; ++u) key[u] = 0;
            for (;;) {
                bool miss = false;
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int q = lane + 32 * u;
                    if (q < G && (unsigned)(key[u] >> STAMP_SHIFT) != want) key[u] = ld_relaxed(&sc->part[kc % COOP_DEPTH][q].stamp);
                }
#pragma unroll
                for (int u = 0; u < PER; ++u)
                    miss |= lane + 32 * u < G && (unsigned)(key[u] >> STAMP_SHIFT) != want;
                if (!__any_sync(0xffffffffu, miss)) break;
                if (__any_sync(0xffffffffu, wb.expired(err))) {
                    ok = false;
                    break;
                }
            }
            // (from here on a failed wait only sets ok: the column runs to its end on
            // whatever was read, with no interchange, and the block leaves after it)
            int W = -1;
            {
                unsigned long long K = 0;
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    key[u] &= KEY_MASK;
                    const int q = lane + 32 * u;
                    if (q < G && key[u] > 0 && (W < 0 || key[u] > K)) { K = key[u]; W = q; }
                }
                warp_best_key(K, W);  // lowest slot among equal keys
                int same = 0;
#pragma unroll
                for (int u = 0; u < PER; ++u) same += (lane + 32 * u < G && key[u] == K) ? 1 : 0;
                same = __reduce_add_sync(0xffffffffu, same);
                if (same > 1) {
                    // equal keys: compare the candidates exactly (lowest row on ties)
                    MPF<L> v = mpf_make_zero<L>();
                    int vi = -1, vw = -1;
#pragma unroll 1
                    for (int u = 0; u < PER; ++u) {
                        const int q = lane + 32 * u;
                        bool mine = false;
#pragma unroll
                        for (int t = 0; t < PER; ++t) mine |= t == u && q < G && key[t] == K;
                        const CoopSlot<L>& slot = sc->part[kc % COOP_DEPTH][mine ? q : 0];
                        const unsigned long long* p[WORDS + 1];
                        uint32_t w[WORDS + 1];
#pragma unroll
                        for (int i = 0; i < WORDS; ++i) p[i] = mine ? &slot.row[i][kc] : nullptr;
                        p[WORDS] = mine ? &slot.idx : nullptr;
                        ok = ok && wait_words<WORDS + 1>(p, tag, w, err);
                        MPF<L> y;
#pragma unroll
                        for (int i = 0; i < L; ++i) y.m[i] = w[i];
                        y.e = (int)w[L];
                        y.neg = (int)w[L + 1];
                        if (mine && mpf_better<L>(y, (int)w[WORDS], v, vi)) { v = y; vi = (int)w[WORDS]; vw = q; }
                    }
                    warp_best<L>(v, vi, vw);
                    W = vw;
                }
                if (W < 0) W = 0;  // (some block has a candidate: row c itself is one)
            }
            if (lane == 0) {
                s_slot = W;
                if (!ok) s_fail[kc & 1] = 1;
            }
            bar_sync(BAR_PIVOT, 128);
            // the pivot's row, its element of column kc + 1, old row c's two
            // elements (for the owner of the pivot row); then the reciprocal
            const CoopSlot<L>& ws = sc->part[kc % COOP_DEPTH][W];
            const bool word = lane < WORDS;
            uint32_t w[4], wr[1];
            {
                const unsigned long long* p[4];
                p[0] = &ws.idx;
                p[1] = word && !last ? &ws.row[word ? lane : 0][last ? kc : kc + 1] : nullptr;
                p[2] = word ? orow + lane * PBASE + kc : nullptr;
                p[3] = word && !last ? orow + lane * PBASE + kc + 1 : nullptr;
                ok &= wait_words<4>(p, tag, w, err);
            }
            const int piv = ok ? (int)w[0] : c;
            const MPF<L> u = mpf_gather<L>(w[1]), ox = mpf_gather<L>(w[2]), oy = mpf_gather<L>(w[3]);
            const bool swapped = piv != c && owns(piv);
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (swapped && lane + 32 * q == piv - r0) x[q] = ox;
            __syncwarp();
            {
                const unsigned long long* p[1] = {word ? &ws.rec[word ? lane : 0] : nullptr};
                ok &= wait_words<1>(p, tag, wr, err);
            }
            const MPF<L> rec = mpf_gather<L>(wr[0]);
            const bool zero = mpf_zero<L>(rec);
            if (!last) {  // the multipliers
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (32 * q < nr) x[q] = mpf_mul<L>(x[q], rec);
            }
            bar_sync(BAR_COL, T);  // column kc + 1 carries the updates up to kc - 1
            if (lane == 0) {
                s_zero = zero ? 1 : 0;
                if (!ok) s_fail[kc & 1] = 1;
            }
            if (!last) {
                MPF<L> y[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    y[q] = mpf_make_zero<L>();
                    if (32 * q >= nr) break;
                    const int r = lane + 32 * q;
                    // (lanes past the last row work on it too, so that the warp stays together)
                    const MPF<L> old = a[min(r, nr - 1) * bs + kc + 1];
                    const bool from = !zero && swapped && r0 + r == piv;
#pragma unroll
                    for (int i = 0; i < L; ++i) y[q].m[i] = from ? oy.m[i] : old.m[i];
                    y[q].e = from ? oy.e : old.e;
                    y[q].neg = from ? oy.neg : old.neg;
                    if (!zero) {
                        y[q] = mpf_fms<L>(y[q], x[q], u);
                        if (r >= lo && r < nr) a[r * bs + kc + 1] = y[q];
                    }
                }
                __syncwarp();
                cand = choose(y, c + 1, kc + 1);
            }
        } else if (warp < 4) {
            bar_sync(BAR_PIVOT, 128);
            const CoopSlot<L>& ws = sc->part[kc % COOP_DEPTH][s_slot];
            if (warp == 1) {
                // the multipliers; the rows' elements of column kc as warp 0 has them
                const bool word = lane < WORDS;
                const unsigned long long* p[3] = {&ws.idx, word ? &ws.rec[word ? lane : 0] : nullptr,
                                                  word ? orow + lane * PBASE + kc : nullptr};
                uint32_t v[3];
                const bool ok = wait_words<3>(p, tag, v, err);
                const int piv = ok ? (int)v[0] : c;
                const MPF<L> rec = mpf_gather<L>(v[1]), ox = mpf_gather<L>(v[2]);
                const bool zero = mpf_zero<L>(rec);
                if (lane == 0) {
                    if (!ok) s_fail[kc & 1] = 1;
                    if (g == 0) {
                        ipiv[c] = piv + 1;
                        if (zero && *info == 0) *info = c + 1;
                    }
                }
                bar_sync(BAR_ROWS, ROWS_T);
                if (!zero)
                    for (int r = lane; r < nr; r += 32)
                        if (r >= lo) a[r * bs + kc] = mpf_mul<L>(piv != c && r0 + r == piv ? ox : a[r * bs + kc], rec);
            } else {
                // the pivot row, and the interchange (the owner of the pivot row
                // leaves columns kc and kc + 1 to warps 1 and 0); two elements a lane
                constexpr int H = PBASE / 64;
                const int k0 = tid - 64;
                const unsigned long long* p[H * WORDS + 2];
                uint32_t v[H * WORDS + 2];
#pragma unroll
                for (int h = 0; h < H; ++h)
#pragma unroll
                    for (int i = 0; i < WORDS; ++i) p[h * WORDS + i] = k0 + 64 * h < b ? &ws.row[i][(k0 + 64 * h) & (PBASE - 1)] : nullptr;
                p[H * WORDS] = &ws.idx;
                p[H * WORDS + 1] = &ws.row[L - 1][kc];  // the pivot's top limb
                bool ok = wait_words<H * WORDS + 2>(p, tag, v, err);
                const int piv = ok ? (int)v[H * WORDS] : c;
                const bool swap = v[H * WORDS + 1] != 0 && piv != c;
                bar_sync(BAR_ROWS, ROWS_T);
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const int k = k0 + 64 * h;
                    MPF<L> e;
#pragma unroll
                    for (int i = 0; i < L; ++i) e.m[i] = v[h * WORDS + i];
                    e.e = (int)v[h * WORDS + L];
                    e.neg = (int)v[h * WORDS + L + 1];
                    if (k < b) {
                        pr[k] = e;
                        if (swap && owns(c)) a[(c - r0) * bs + k] = e;
                    }
                }
                if (swap && owns(piv)) {
#pragma unroll
                    for (int h = 0; h < H; ++h)
#pragma unroll
                        for (int i = 0; i < WORDS; ++i)
                            p[h * WORDS + i] = k0 + 64 * h < b ? orow + i * PBASE + ((k0 + 64 * h) & (PBASE - 1)) : nullptr;
                    p[H * WORDS] = nullptr;
                    p[H * WORDS + 1] = nullptr;
                    ok &= wait_words<H * WORDS + 2>(p, tag, v, err);
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        const int k = k0 + 64 * h;
                        MPF<L> e;
#pragma unroll
                        for (int i = 0; i < L; ++i) e.m[i] = v[h * WORDS + i];
                        e.e = (int)v[h * WORDS + L];
                        e.neg = (int)v[h * WORDS + L + 1];
                        if (k < b && k != kc && k != kc + 1) a[(piv - r0) * bs + k] = e;
                    }
                }
                if (!ok && lane == 0) s_fail[kc & 1] = 1;
            }
        } else if (bulk_kc >= 0) {
            // warps 4 ..: the deferred update of the other rows by column bulk_kc
            // (from bulk_kc + 3 on: warp 1 took column bulk_kc + 2)
            const int kb = bulk_kc, rest = b - kb - 3;
            const MPF<L>* pk = prow[kb & 1];
            const int total = rest > 0 ? (nr - bulk_lo) * rest : 0;
            for (int p = tid - 128; p < total; p += T - 128) {
                const int r = bulk_lo + p / rest, k = kb + 3 + (p - (p / rest) * rest);
                if (r == bulk_pa || r == bulk_pb) continue;
                a[r * bs + k] = mpf_fms_oolv<L>(a[r * bs + k], a[r * bs + kb], pk[k]);
            }
        }
        __syncthreads();
        if (s_fail[kc & 1]) return;
        if (last) break;
        const bool zero = s_zero != 0;
        const int pa = s_cand >= 0 ? s_cand - r0 : -1;
        const int pb = owns(c + 1) ? c + 1 - r0 : -1;
        if (warp == 0) {
            publish_rec(cand, kc + 1);
        } else {
            if (pub >= 0) {
                publish_rows(kc, zero, pa, pb);
                bar_arrive(BAR_ROWS, ROWS_T);
            } else if (warp == 1 && !zero && kc + 2 < b) {
                for (int r = lo + lane; r < nr; r += 32)
                    if (r != pa && r != pb)
                        a[r * bs + kc + 2] = mpf_fms_oolv<L>(a[r * bs + kc + 2], a[r * bs + kc], pr[kc + 2]);
            }
            bar_arrive(BAR_COL, T);
        }
        bulk_kc = zero ? -1 : kc;
        bulk_lo = lo;
        bulk_pa = pa;
        bulk_pb = pb;
    }
    for (int p = tid; p < nr * b; p += T) {
        const int r = p / b, k = p - r * b;
        mpf_to_exp<L, N>(a[r * bs + k], elem(A, lda, N, r0 + r, c0 + k));
    }
}

}  // namespace
}  // namespace ozlu
