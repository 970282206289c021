// Blocked right-looking LU with partial pivoting and the solve (Sec. 3.4).
//
//   for each panel of width nb:
//     (P1) factor the n - r0 by nb panel: recursive halving down to base
//          blocks of BASE columns; a base block is factored column by column
//          in expansion arithmetic (pivot search, interchange across the
//          panel, scaling, rank-1 update of the base block); between halves
//          U12 = L11^-1 A12 by a recursive triangular solve and
//          A22 -= L21 U12 by the Ozaki-II GEMM;
//     (P2) apply the interchanges to the columns left and right of the panel;
//     (P3) U12 = L11^-1 A12, recursive triangular solve;
//     (P4) A22 <- A22 - L21 U12 (Eq. (13)) by the Ozaki-II GEMM.
// Only (P4) is the update the paper moves to Ozaki scheme II; the recursion
// puts the larger part of (P1) and (P3) on the same GEMM as well, leaving
// O(n^2 BASE) operations in FP64 expansion arithmetic (the GB300 FP64 rate is
// about 1 TFLOP/s).  getrs: interchanges, then forward (unit L)
// and backward (U) substitution: for a few right-hand sides each as one
// cooperative kernel in multi-limb floats, else blocked, with base triangles in
// them and the off-diagonal updates by the Ozaki-II GEMM.
#include <string.h>

#include <tuple>

#include "launch.cuh"
#include "expansion.cuh"
#include "mpf.cuh"
#include "ozlu_handle.h"
#include "panel.cuh"

namespace ozlu {
namespace {

constexpr int BASE = 32;        // triangular-solve leaves and the fallback panel path
constexpr int PIV_THREADS = 256;
constexpr int PIV_BLOCKS = 152;
constexpr int MAXPART = 1024;   // block partials of a column step
constexpr int STEP_ROWS = 16;   // rows per block of a column step
constexpr int TRSM_WARPS = 16;  // columns per block of a base triangular solve, at most
constexpr int LCT = 4;          // laswp: columns per block
constexpr int LMAXB = 512;      // laswp: interchanges per call
constexpr int TRI_SLOTS = 8;    // triangles of base solves converted ahead (256 / BASE)

struct LuScratch {
    uint32_t rm[8];             // reciprocal of the current pivot (MPF words)
    int re, rneg;
    int piv;
    int zero;
    unsigned int counter;
    int info;
    int result;                 // info as reported by ozlu_getrf (finish_kernel)
    double pval[MAXPART][4];    // block candidates (expansion values)
    int pidx[MAXPART];
    int plist[1 + 4 * LMAXB];   // interchange permutation: count, (dst, src) pairs
    // triangles of base triangular solves as L-limb floats: [k][i], then the
    // reciprocal diagonal (upper case); slot q holds the q-th diagonal block of
    // a unit lower triangle converted ahead of its recursion
    alignas(16) unsigned char tri[TRI_SLOTS][(BASE * BASE + BASE) * sizeof(MPF<8>)];
};

template <int L>
__device__ __forceinline__ void put_recip(LuScratch* sc, const MPF<L>& r) {
#pragma unroll
    for (int i = 0; i < L; ++i) sc->rm[i] = r.m[i];
    sc->re = r.e;
    sc->rneg = r.neg;
}

template <int L>
__device__ __forceinline__ MPF<L> get_recip(const LuScratch* sc) {
    MPF<L> r;
#pragma unroll
    for (int i = 0; i < L; ++i) r.m[i] = sc->rm[i];
    r.e = sc->re;
    r.neg = sc->rneg;
    return r;
}

// better(a, ia, b, ib): |a| > |b|, or equal and ia < ib (first index on ties)
template <int N>
__device__ __forceinline__ bool better(const Exp<N>& a, int ia, const Exp<N>& b, int ib) {
    if (ib < 0) return ia >= 0;
    if (ia < 0) return false;
    const int c = abs_cmp<N>(a, b);
    return c > 0 || (c == 0 && ia < ib);
}

// Last-block reduction of the block candidates: each thread scans a strided
// share of the partials, then a shared-memory tree keeps the best (largest
// magnitude, first index on ties).  All threads of the block must call it;
// the result is valid in thread 0.
template <int N, int THREADS>
__device__ __forceinline__ void reduce_partials(const LuScratch* sc, int nparts, Exp<N>& b, int& ib) {
    __shared__ double rv[THREADS][N];
    __shared__ int ri[THREADS];
    Exp<N> best;
    int bi = -1;
#pragma unroll
    for (int q = 0; q < N; ++q) best.x[q] = 0.0;
    for (int k = threadIdx.x; k < nparts; k += THREADS) {
        Exp<N> v;
#pragma unroll
        for (int q = 0; q < N; ++q) v.x[q] = ((volatile const double*)sc->pval[k])[q];
        const int iv = ((volatile const int*)sc->pidx)[k];
        if (better<N>(v, iv, best, bi)) { best = v; bi = iv; }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) rv[threadIdx.x][q] = best.x[q];
    ri[threadIdx.x] = bi;
    __syncthreads();
    for (int s = THREADS / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            Exp<N> u, v;
#pragma unroll
            for (int q = 0; q < N; ++q) { u.x[q] = rv[threadIdx.x][q]; v.x[q] = rv[threadIdx.x + s][q]; }
            if (better<N>(v, ri[threadIdx.x + s], u, ri[threadIdx.x])) {
#pragma unroll
                for (int q = 0; q < N; ++q) rv[threadIdx.x][q] = v.x[q];
                ri[threadIdx.x] = ri[threadIdx.x + s];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < N; ++q) b.x[q] = rv[0][q];
    ib = ri[0];
}

// Pivot search of column c over rows [c, n); the last block to finish reduces
// the block results, interchanges rows c and piv over columns [p0, p1),
// records ipiv[c] (1-based) and the reciprocal of the pivot.
template <int N>
__global__ void __launch_bounds__(PIV_THREADS) pivot_kernel(double* A, long long lda, int n, int c,
                                                            int p0, int p1, int* ipiv,
                                                            LuScratch* sc) {
    chain_enter();
    __shared__ double sv[PIV_THREADS][N];
    __shared__ int si[PIV_THREADS];
    __shared__ bool last;
    Exp<N> best;
    int bi = -1;
#pragma unroll
    for (int q = 0; q < N; ++q) best.x[q] = 0.0;
    for (int i = c + blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        Exp<N> v = load<N>(elem(A, lda, N, i, c));
        if (better<N>(v, i, best, bi)) { best = v; bi = i; }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) sv[threadIdx.x][q] = best.x[q];
    si[threadIdx.x] = bi;
    __syncthreads();
    for (int s = PIV_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            Exp<N> a, b;
#pragma unroll
            for (int q = 0; q < N; ++q) { a.x[q] = sv[threadIdx.x][q]; b.x[q] = sv[threadIdx.x + s][q]; }
            if (better<N>(b, si[threadIdx.x + s], a, si[threadIdx.x])) {
#pragma unroll
                for (int q = 0; q < N; ++q) sv[threadIdx.x][q] = b.x[q];
                si[threadIdx.x] = si[threadIdx.x + s];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < N; ++q) sc->pval[blockIdx.x][q] = sv[0][q];
        sc->pidx[blockIdx.x] = si[0];
        __threadfence();
        const unsigned int done = atomicAdd(&sc->counter, 1u);
        last = done == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    __shared__ int piv;
    Exp<N> b;
    int ib;
    reduce_partials<N, PIV_THREADS>(sc, gridDim.x, b, ib);
    if (threadIdx.x == 0) {
        if (ib < 0) ib = c;
        piv = ib;
        sc->piv = ib;
        ipiv[c] = ib + 1;
        sc->counter = 0;
        const bool zero = b.x[0] == 0.0;
        sc->zero = zero ? 1 : 0;
        if (zero && sc->info == 0) sc->info = c + 1;
        if (!zero) {
            constexpr int L = Limbs<N>::L;
            put_recip<L>(sc, mpf_recip<L>(mpf_from_exp<L, N>(b.x)));
        }
    }
    __syncthreads();
    const int pv = piv;
    if (pv != c) {
        for (int j = p0 + threadIdx.x; j < p1; j += blockDim.x) {
            double* a = elem(A, lda, N, c, j);
            double* b = elem(A, lda, N, pv, j);
#pragma unroll
            for (int q = 0; q < N; ++q) { const double t = a[q]; a[q] = b[q]; b[q] = t; }
        }
    }
}

// One column step of a base block, fused with the next pivot search.
// Rows i in (c, n): l_i = a_ic * (1 / pivot), a_ik -= l_i a_ck for k in (c, c1),
// all in L-limb integer floating point; each block then offers its best
// candidate for column c + 1 and the last block to finish reduces them,
// interchanges rows c + 1 and piv over the outer panel columns [p0, p1),
// records ipiv and the reciprocal of the new pivot.
template <int N>
__global__ void __launch_bounds__(128) column_step_kernel(double* A, long long lda, int n, int c,
                                                          int c1, int p0, int p1, int* ipiv,
                                                          LuScratch* sc) {
    chain_enter();
    constexpr int L = Limbs<N>::L;
    __shared__ MPF<L> urow[BASE];
    __shared__ MPF<L> lrow[STEP_ROWS];
    __shared__ double cand[STEP_ROWS][N];
    __shared__ int candi[STEP_ROWS];
    __shared__ bool last;
    __shared__ int piv;
    const int cols = c1 - c - 1;
    const bool zero = sc->zero != 0;
    for (int k = threadIdx.x; k < cols; k += blockDim.x)
        urow[k] = mpf_from_exp<L, N>(elem(A, lda, N, c, c + 1 + k));
    // candidate of this thread (threads < STEP_ROWS) over its rows of all chunks
    Exp<N> best;
    int bi = -1;
#pragma unroll
    for (int q = 0; q < N; ++q) best.x[q] = 0.0;
    const int nchunks = (n - c - 1 + STEP_ROWS - 1) / STEP_ROWS;
    for (int chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
        const int i0 = c + 1 + chunk * STEP_ROWS;
        __syncthreads();
        if (threadIdx.x < STEP_ROWS) {
            const int i = i0 + threadIdx.x;
            if (i < n && !zero) {
                double* ai = elem(A, lda, N, i, c);
                MPF<L> l = mpf_mul<L>(mpf_from_exp<L, N>(ai), get_recip<L>(sc));
                mpf_to_exp<L, N>(l, ai);
                lrow[threadIdx.x] = l;
            }
        }
        __syncthreads();
        if (!zero) {
            for (int pidx = threadIdx.x; pidx < STEP_ROWS * cols; pidx += blockDim.x) {
                const int k = pidx / STEP_ROWS, rr = pidx - k * STEP_ROWS;
                const int i = i0 + rr;
                if (i >= n) continue;
                double* a = elem(A, lda, N, i, c + 1 + k);
                mpf_to_exp<L, N>(mpf_fms<L>(mpf_from_exp<L, N>(a), lrow[rr], urow[k]), a);
            }
        }
        if (cols > 0) {
            __syncthreads();
            if (threadIdx.x < STEP_ROWS) {
                const int i = i0 + threadIdx.x;
                if (i < n) {
                    const Exp<N> v = load<N>(elem(A, lda, N, i, c + 1));
                    if (better<N>(v, i, best, bi)) { best = v; bi = i; }
                }
            }
        }
    }
    if (cols == 0) return;  // last column of the base block: no next pivot here
    if (threadIdx.x < STEP_ROWS) {
#pragma unroll
        for (int q = 0; q < N; ++q) cand[threadIdx.x][q] = best.x[q];
        candi[threadIdx.x] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Exp<N> b;
        int ib = -1;
#pragma unroll
        for (int q = 0; q < N; ++q) b.x[q] = 0.0;
        for (int r = 0; r < STEP_ROWS; ++r) {
            Exp<N> v;
#pragma unroll
            for (int q = 0; q < N; ++q) v.x[q] = cand[r][q];
            if (better<N>(v, candi[r], b, ib)) { b = v; ib = candi[r]; }
        }
#pragma unroll
        for (int q = 0; q < N; ++q) sc->pval[blockIdx.x][q] = b.x[q];
        sc->pidx[blockIdx.x] = ib;
        __threadfence();
        const unsigned int done = atomicAdd(&sc->counter, 1u);
        last = done == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int cn = c + 1;
    Exp<N> b;
    int ib;
    reduce_partials<N, 128>(sc, gridDim.x, b, ib);
    if (threadIdx.x == 0) {
        if (ib < 0) ib = cn;
        piv = ib;
        ipiv[cn] = ib + 1;
        sc->counter = 0;
        const bool z = b.x[0] == 0.0;
        sc->zero = z ? 1 : 0;
        if (z && sc->info == 0) sc->info = cn + 1;
        if (!z) put_recip<L>(sc, mpf_recip<L>(mpf_from_exp<L, N>(b.x)));
    }
    __syncthreads();
    const int pv = piv;
    if (pv != cn) {
        for (int j = p0 + threadIdx.x; j < p1; j += blockDim.x) {
            double* a = elem(A, lda, N, cn, j);
            double* b = elem(A, lda, N, pv, j);
#pragma unroll
            for (int q = 0; q < N; ++q) { const double t = a[q]; a[q] = b[q]; b[q] = t; }
        }
    }
}

// the error word and every tagged word of G slots start at zero for each
// factorisation (grid G x COOP_DEPTH; the scratch was laid out for L limbs)
template <int L>
__global__ void coop_reset_kernel(CoopScratch<L>* sc) {
    unsigned long long* w = reinterpret_cast<unsigned long long*>(&sc->part[blockIdx.y][blockIdx.x]);
    for (int t = threadIdx.x; t < (int)(sizeof(CoopSlot<L>) / 8); t += blockDim.x) w[t] = 0ull;
    if (blockIdx.x == 0) {
        unsigned long long* o = &sc->orow[blockIdx.y][0][0];
        for (int t = threadIdx.x; t < (L + 2) * PBASE; t += blockDim.x) o[t] = 0ull;
        if (blockIdx.y == 0 && threadIdx.x == 0) sc->error = 0;
    }
}

// Apply interchanges k in [k0, k1) (ipiv 1-based) to columns [j0, j1).
template <int N>
__global__ void laswp_kernel(double* A, long long lda, int j0, int j1, int k0, int k1,
                             const int* ipiv) {
    chain_enter();
    const int j = j0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= j1) return;
    for (int k = k0; k < k1; ++k) {
        const int p = ipiv[k] - 1;
        if (p != k) {
            double* a = elem(A, lda, N, k, j);
            double* b = elem(A, lda, N, p, j);
#pragma unroll
            for (int q = 0; q < N; ++q) { const double t = a[q]; a[q] = b[q]; b[q] = t; }
        }
    }
}

// Interchanges k in [k0, k1) (ipiv 1-based) applied to columns [j0, j1) as one
// permutation: one block lists the (destination, source) row pairs, then every
// block of laswp_apply_kernel gathers those rows of its LCT columns into shared
// memory and writes them back permuted.  Replaces the column-serial swap chain.

// Position k < b stands for row k0 + k, position b + j for a row p >= k1 first
// named by interchange j.  The threads find each interchange's positions; one
// thread then replays the swaps on the contents (two shared-memory loads and
// stores a swap, the next positions loaded ahead).  With a hash map filled by that
// thread the list took 50 us for 256 interchanges.
__global__ void __launch_bounds__(LMAXB) laswp_list_kernel(int k0, int k1, const int* ipiv, int* list) {
    chain_enter();
    __shared__ int piv[LMAXB], slot[LMAXB + 1], val[2 * LMAXB], row[2 * LMAXB];
    __shared__ int cnt;
    const int b = k1 - k0, t = threadIdx.x;
    if (t < b) piv[t] = ipiv[k0 + t] - 1;
    if (t == 0) cnt = 0;
    __syncthreads();
    if (t < b) {
        const int p = piv[t];
        const bool out = p < k0 || p >= k1;
        int j = t;
        if (out)
            for (j = 0; piv[j] != p; ++j) {}
        slot[t] = out ? b + j : p - k0;
        row[t] = val[t] = k0 + t;
        row[b + t] = out && j == t ? p : -1;
        val[b + t] = p;
    }
    __syncthreads();
    if (t == 0) {
        int nxt = slot[0];
        for (int k = 0; k < b; ++k) {
            const int sl = nxt;
            nxt = slot[k + 1];  // (one past the end is in bounds)
            const int x = val[k], y = val[sl];
            val[k] = y;
            val[sl] = x;
        }
    }
    __syncthreads();
    for (int q = t; q < 2 * b; q += blockDim.x)
        if (row[q] >= 0 && val[q] != row[q]) {
            const int c = atomicAdd(&cnt, 1);
            list[1 + 2 * c] = row[q];
            list[2 + 2 * c] = val[q];
        }
    __syncthreads();
    if (t == 0) list[0] = cnt;
}

template <int N>
__global__ void __launch_bounds__(256) laswp_apply_kernel(double* A, long long lda, int j0, int j1,
                                                          const int* list) {
    chain_enter();
    extern __shared__ __align__(16) double buf[];  // [entry][col][N]
    const int ne = list[0];
    const int jb = j0 + blockIdx.x * LCT;
    for (int t = threadIdx.x; t < ne * LCT; t += blockDim.x) {
        const int e = t / LCT, cc = t - e * LCT, j = jb + cc;
        if (j < j1) {
            const double* x = elem(A, lda, N, list[2 + 2 * e], j);
#pragma unroll
            for (int q = 0; q < N; ++q) buf[(e * LCT + cc) * N + q] = x[q];
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < ne * LCT; t += blockDim.x) {
        const int e = t / LCT, cc = t - e * LCT, j = jb + cc;
        if (j < j1) {
            double* x = elem(A, lda, N, list[1 + 2 * e], j);
#pragma unroll
            for (int q = 0; q < N; ++q) x[q] = buf[(e * LCT + cc) * N + q];
        }
    }
}

// the permutation of interchanges [k0, k1) applied to column ranges
template <int N>
void laswp2(double* A, long long lda, int ja0, int ja1, int jb0, int jb1, int k0, int k1, const int* ipiv,
            int* list, cudaStream_t s) {
    if (k1 <= k0 || (ja1 <= ja0 && jb1 <= jb0)) return;
    if (k1 - k0 > LMAXB) {
        if (ja1 > ja0) launch(laswp_kernel<N>, (ja1 - ja0 + 127) / 128, 128, 0, s, A, lda, ja0, ja1, k0, k1, ipiv);
        if (jb1 > jb0) launch(laswp_kernel<N>, (jb1 - jb0 + 127) / 128, 128, 0, s, A, lda, jb0, jb1, k0, k1, ipiv);
        return;
    }
    launch(laswp_list_kernel, 1, (k1 - k0 + 31) / 32 * 32, 0, s, k0, k1, ipiv, list);
    const size_t smem = sizeof(double) * 2 * (k1 - k0) * LCT * N;
    raise_smem_limit((const void*)laswp_apply_kernel<N>, (int)(sizeof(double) * 2 * LMAXB * LCT * N));
    if (ja1 > ja0) launch(laswp_apply_kernel<N>, (ja1 - ja0 + LCT - 1) / LCT, 256, smem, s, A, lda, ja0, ja1, list);
    if (jb1 > jb0) launch(laswp_apply_kernel<N>, (jb1 - jb0 + LCT - 1) / LCT, 256, smem, s, A, lda, jb0, jb1, list);
}

// Native trailing update for the blocked-naive comparison (Sec. 3.4):
// C -= A B with every multiply-add rounded in expansion arithmetic (binary64
// TwoSum / TwoProd), 16 x 16 outputs per block, A and B tiles in shared memory.
template <int N>
__global__ void __launch_bounds__(256) naive_update_kernel(const double* A, long long lda, const double* B,
                                                           long long ldb, double* C, long long ldc, int m,
                                                           int n, int k) {
    chain_enter();
    __shared__ double sa[16][16][N];
    __shared__ double sb[16][16][N];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i = blockIdx.x * 16 + tx, j = blockIdx.y * 16 + ty;
    Exp<N> acc;
    if (i < m && j < n) acc = load<N>(C + ((long long)i + (long long)j * ldc) * N);
    for (int h0 = 0; h0 < k; h0 += 16) {
        {
            const int ii = blockIdx.x * 16 + tx, hh = h0 + ty;
#pragma unroll
            for (int q = 0; q < N; ++q)
                sa[ty][tx][q] = (ii < m && hh < k) ? A[((long long)ii + (long long)hh * lda) * N + q] : 0.0;
            const int hb = h0 + tx, jj = blockIdx.y * 16 + ty;
#pragma unroll
            for (int q = 0; q < N; ++q)
                sb[ty][tx][q] = (hb < k && jj < n) ? B[((long long)hb + (long long)jj * ldb) * N + q] : 0.0;
        }
        __syncthreads();
        if (i < m && j < n) {
            const int hmax = min(16, k - h0);
            for (int h = 0; h < hmax; ++h) {
                Exp<N> a, b;
#pragma unroll
                for (int q = 0; q < N; ++q) { a.x[q] = sa[h][tx][q]; b.x[q] = sb[ty][h][q]; }
                acc = fms<N>(acc, a, b);
            }
        }
        __syncthreads();
    }
    if (i < m && j < n) store<N>(C + ((long long)i + (long long)j * ldc) * N, acc);
}

// The b x b triangle of a base triangular solve, converted once to L-limb
// floats (and the reciprocal diagonal for the upper case) in the scratch:
// blockIdx.y = q converts the q-th b x b diagonal block from T into slot q.
template <int N>
__global__ void __launch_bounds__(256) tri_convert_kernel(const double* T, long long ldt, int b, int lower,
                                                          LuScratch* sc) {
    chain_enter();
    constexpr int L = Limbs<N>::L;
    const int q = blockIdx.y;
    T += ((long long)q * b + (long long)q * b * ldt) * N;
    MPF<L>* tl = reinterpret_cast<MPF<L>*>(sc->tri[q]);
    MPF<L>* rd = tl + BASE * BASE;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < b * b; idx += gridDim.x * blockDim.x) {
        const int i = idx / b, k = idx - i * b;
        const bool need = lower ? (k < i) : (k >= i);
        const MPF<L> v = need ? mpf_from_exp<L, N>(T + ((long long)i + (long long)k * ldt) * N) : mpf_make_zero<L>();
        tl[k * BASE + i] = v;  // column-major: a step reads one column across the rows
        if (!lower && i == k) rd[k] = mpf_zero<L>(v) ? mpf_make_zero<L>() : mpf_recip<L>(v);
    }
}

// X <- L^-1 X for a unit lower (lower = 1) or U^-1 X for an upper (lower = 0,
// non-unit) b x b triangle, b <= BASE; X is b x ncols.  L-limb integer
// floating point.  One warp per column, lane i holding x_i in registers: step
// k broadcasts the final x_k by warp shuffles and every lane below (lower) or
// above (upper) row k subtracts l_ik x_k, so the b steps need no block-wide
// barrier and the warps of a block progress independently.  The triangle comes
// to shared memory by asynchronous copies while X is converted, and is read
// column by column ([k][i], conflict-free).  The warps stay converged (every
// lane multiplies and selects).
template <int N>
__global__ void __launch_bounds__(TRSM_WARPS * 32) trsm_base_kernel(const LuScratch* sc, double* X, long long ldx,
                                                                    int b, int ncols, int lower, int slot) {
    chain_enter();
    constexpr int L = Limbs<N>::L;
    extern __shared__ __align__(16) unsigned char smraw[];
    MPF<L>* sl = reinterpret_cast<MPF<L>*>(smraw);   // [k][i]
    MPF<L>* rd = sl + BASE * BASE;                   // reciprocal diagonal (upper)
    const int row = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int col = blockIdx.x * (blockDim.x >> 5) + w;
    constexpr int CHUNKS = (BASE * BASE + BASE) * (int)sizeof(MPF<L>) / 16;
    static_assert((BASE * BASE + BASE) * sizeof(MPF<L>) % 16 == 0, "whole 16-byte pieces");
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smraw);
    for (int i = threadIdx.x; i < CHUNKS; i += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(sc->tri[slot] + 16 * i)
                     : "memory");
    const bool mine = row < b && col < ncols;
    double* xp = X + ((long long)row + (long long)col * ldx) * N;
    MPF<L> x = mine ? mpf_from_exp<L, N>(xp) : mpf_make_zero<L>();
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
#pragma unroll 1
    for (int s = 0; s < b; ++s) {
        const int k = lower ? s : b - 1 - s;
        if (!lower) {
            const MPF<L> v = mpf_mul<L>(x, rd[k]);
            mpf_take<L>(x, v, row == k);
        }
        const MPF<L> v = mpf_fms<L>(x, sl[k * BASE + row], mpf_bcast<L>(x, k));
        mpf_take<L>(x, v, lower ? row > k : row < k);
    }
    if (mine) mpf_to_exp<L, N>(x, xp);
}

// slot < 0: convert the triangle into slot 0 first; else it is in `slot`
template <int N>
void trsm_base(const double* T, long long ldt, double* X, long long ldx, int b, int ncols, int lower,
               LuScratch* sc, cudaStream_t s, int slot = -1) {
    if (ncols <= 0 || b <= 0) return;
    constexpr int L = Limbs<N>::L;
    if (slot < 0) {
        launch(tri_convert_kernel<N>, (b * b + 255) / 256, 256, 0, s, T, ldt, b, lower, sc);
        slot = 0;
    }
    // every SM the same number of columns: blocks of equal size, one or two an SM
    const int sms = device_sms(), per = (ncols + TRSM_WARPS * sms - 1) / (TRSM_WARPS * sms) * sms;
    const int wpb = (ncols + per - 1) / per;
    const size_t smem = sizeof(MPF<L>) * (BASE * BASE + BASE);
    raise_smem_limit((const void*)trsm_base_kernel<N>, (int)smem);
    launch(trsm_base_kernel<N>, (ncols + wpb - 1) / wpb, 32 * wpb, smem, s, sc, X, ldx, b, ncols, lower, slot);
}

// ---------------------------------------------------------------------------
// X <- L^-1 X (unit lower) or U^-1 X for a few right-hand sides as one
// cooperative kernel per direction.  A block owns 32 rows (block-rows t = g,
// g + G, ... in the order of the substitution): it subtracts the products with
// every earlier x as it is announced, then solves its triangle and announces its
// own rows, SOLVE_PART at a time, as tagged words (as the panel kernel does).
// Everything is in L-limb floats, X rounded to expansions once per direction.
//   lane = row; the 16 warps are KW parts of k times the right-hand sides
//   (KW = 16 / the power of two >= nrhs), each with a partial sum of its own
//   over all blocks, added once at the end in a fixed order.
// Bound by latency: of the 24 us (QD) a block-row takes, 19 are its 32 dependent
// multiply-subtracts (about 1170 cycles each with the broadcast), 3 the last
// part of x_{t-1} on all warps and 2 the sum of the parts.  The products with
// all other x and the conversion of the next 32 x 32 factors (SOLVE_BUF buffers)
// run ahead of the chain.  The warps that solve the triangle, one a right-hand
// side, issue from different schedulers: on one, three took 1940 cycles a step.
// The upper triangle is scaled by the reciprocals of its diagonal beforehand (a
// zero pivot gives 0), so that both directions have unit steps.
// The other form, kept above SOLVE_RHS: base triangles of 32 rows and an Ozaki-II
// GEMM after each, its time hardly depending on nrhs.  Milliseconds, here / there,
// for 1, 8, 9 and 16 right-hand sides:
//   QD n =   256   0.42 / 0.81   0.58 / 0.82   0.78 / 0.83   0.96 / 0.83
//      n =  1024   1.6 / 3.6     2.2 / 3.6     3.2 / 3.6     3.9 / 3.6
//      n =  4096   5.7 / 17.9    8.2 / 18.1   11.4 / 18.1   14.3 / 18.5
//      n = 16384  22.8 / 130    51 / 133      75 / 134      94 / 140
//   DD n =   256   0.31 / 0.59   0.39 / 0.59   0.52 / 0.59   0.62 / 0.60
//      n =  4096   4.1 / 12.2    5.3 / 12.3    7.3 / 12.3    8.9 / 12.6
// so 13 to 16 lose up to a sixth below n = 1500 or so.  They take it all the same:
// X is rounded to expansions once per direction, not after every 32 rows, and the
// mean error is 3 to 50 times smaller (n = 60 to 1500), the largest one too.  Two
// rounds of 16 would be slower than the other form.
constexpr int SOLVE_RHS = 16;
constexpr int SOLVE_BUF = 3;
constexpr int SOLVE_PART = 8;  // rows announced together

template <int L>
size_t solve_smem(int nrhs) {
    return sizeof(MPF<L>) * (SOLVE_BUF * BASE * BASE + BASE * BASE + BASE + 16 * 32 + (size_t)SOLVE_BUF * nrhs * BASE);
}

template <int N, bool LOWER>
__global__ void __launch_bounds__(512, 1) solve_kernel(const double* T, long long ldt, int n, double* X, long long ldx,
                                                       int nrhs, int kw, unsigned long long* words, int* err) {
    constexpr int L = Limbs<N>::L, WORDS = L + 2;
    extern __shared__ __align__(16) unsigned char smraw[];
    MPF<L>* lb = reinterpret_cast<MPF<L>*>(smraw);    // [SOLVE_BUF][k][i]
    MPF<L>* tri = lb + SOLVE_BUF * BASE * BASE;       // [k][i]
    MPF<L>* rd = tri + BASE * BASE;                   // reciprocal diagonal (upper)
    MPF<L>* part = rd + BASE;                         // [warp][row]
    MPF<L>* xs = part + 16 * 32;                      // [SOLVE_BUF][j][k]
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int nb = (n + BASE - 1) / BASE, G = gridDim.x;
    // right-hand side, part of k: the warps of one part issue from different schedulers
    const int nj = 16 / kw, kp = warp / nj, j = warp - kp * nj;
    auto row0 = [&](int t) { return (LOWER ? t : nb - 1 - t) * BASE; };
    // factors of block-row t against block-column s (both in solve order) into a buffer
    auto convert = [&](int t, int s, int buf) {
        const int i = row0(t) + lane, c0 = row0(s);
#pragma unroll 1
        for (int k = warp; k < BASE; k += 16) {
            MPF<L> v = mpf_make_zero<L>();
            if (i < n && c0 + k < n) v = mpf_from_exp<L, N>(T + ((long long)i + (long long)(c0 + k) * ldt) * N);
            lb[(buf * BASE + k) * BASE + lane] = v;
        }
    };
    for (int t = blockIdx.x; t < nb; t += G) {
        const int i0 = row0(t), bi = min(BASE, n - i0);
        __syncthreads();
        if (!LOWER) {
            if (tid < BASE) {
                MPF<L> d = mpf_make_zero<L>();
                if (tid < bi) d = mpf_from_exp<L, N>(T + ((long long)(i0 + tid) + (long long)(i0 + tid) * ldt) * N);
                rd[tid] = mpf_zero<L>(d) ? mpf_make_zero<L>() : mpf_recip<L>(d);
            }
            __syncthreads();
        }
        for (int k = warp; k < BASE; k += 16) {
            MPF<L> v = mpf_make_zero<L>();
            if (lane < bi && k < bi && (LOWER ? k < lane : k > lane)) {
                v = mpf_from_exp<L, N>(T + ((long long)(i0 + lane) + (long long)(i0 + k) * ldt) * N);
                if (!LOWER) v = mpf_mul<L>(v, rd[lane]);
            }
            tri[k * BASE + lane] = v;
        }
        MPF<L> acc = mpf_make_zero<L>();
        if (kp == 0 && j < nrhs && lane < bi)
            acc = mpf_from_exp<L, N>(X + ((long long)(i0 + lane) + (long long)j * ldx) * N);
        if (t > 0) convert(t, 0, 0);
        for (int s = 0; s < t; ++s) {
            const int buf = s % SOLVE_BUF;
            if (s + 1 < t) convert(t, s + 1, (s + 1) % SOLVE_BUF);
            const unsigned long long* w = words + (size_t)s * nrhs * WORDS * BASE;
            // the newest x in the parts in which it is announced, older ones whole
            const int parts = s == t - 1 ? BASE / SOLVE_PART : 1, len = BASE / parts;
            for (int g = 0; g < parts; ++g) {
                const int k0 = LOWER ? g * len : BASE - (g + 1) * len;
                WaitBound wb;
                for (int q = tid; q < nrhs * WORDS * len; q += 512) {
                    const int k = k0 + q % len, r = q / len;  // r = right-hand side x word
                    unsigned long long v = ld_relaxed(w + r * BASE + k);
                    while ((unsigned)(v >> 32) != 1u) {
                        if (wb.expired(err)) break;  // then the rest is soon done, with wrong numbers
                        if (s + 2 < t) __nanosleep(500);  // not next in the chain: keep off the L2 lines
                        v = ld_relaxed(w + r * BASE + k);
                    }
                    reinterpret_cast<uint32_t*>(&xs[(buf * nrhs + r / WORDS) * BASE + k])[r % WORDS] = (uint32_t)v;
                }
                __syncthreads();
                if (j < nrhs)
                    for (int k = k0 + kp; k < k0 + len; k += kw)
                        acc = mpf_fms<L>(acc, lb[(buf * BASE + k) * BASE + lane], xs[(buf * nrhs + j) * BASE + k]);
            }
        }
        // the partial sums of a right-hand side, pairwise
        part[warp * 32 + lane] = acc;
        for (int o = 1; o < kw; o *= 2) {
            __syncthreads();
            if ((kp & (2 * o - 1)) == 0) {
                acc = mpf_add<L>(acc, part[(warp + o * nj) * 32 + lane]);
                part[warp * 32 + lane] = acc;
            }
        }
        __syncthreads();
        if (kp == 0 && j < nrhs) {
            MPF<L> x = acc;
            if (!LOWER) x = mpf_mul<L>(x, rd[lane]);
            unsigned long long* w = words + ((size_t)t * nrhs + j) * WORDS * BASE;
            // (every lane multiplies and selects: a branch would cost more than it saves)
            for (int g = 0; g < BASE / SOLVE_PART; ++g) {
                const int first = LOWER ? g * SOLVE_PART : BASE - 1 - g * SOLVE_PART;
#pragma unroll 1
                for (int q = 0; q < SOLVE_PART; ++q) {
                    const int k = LOWER ? first + q : first - q;
                    const MPF<L> v = mpf_fms<L>(x, tri[k * BASE + lane], mpf_bcast<L>(x, k));
                    mpf_take<L>(x, v, LOWER ? lane > k : lane < k);
                }
                if ((LOWER ? lane - first : first - lane) >= 0 && (LOWER ? lane - first : first - lane) < SOLVE_PART)
#pragma unroll
                    for (int i = 0; i < WORDS; ++i) st_relaxed(w + i * BASE + lane, (1ull << 32) | mpf_word<L>(x, i));
            }
            if (lane < bi) mpf_to_exp<L, N>(x, X + ((long long)(i0 + lane) + (long long)j * ldx) * N);
        }
    }
}

// interchanges k in [0, n) on the right-hand sides, LMAXB at a time
template <int N>
void laswp_all(double* B, long long ldb, int nrhs, int n, const int* ipiv, int* list, cudaStream_t s) {
    for (int k0 = 0; k0 < n; k0 += LMAXB) laswp2<N>(B, ldb, 0, nrhs, 0, 0, k0, k0 + LMAXB < n ? k0 + LMAXB : n, ipiv, list, s);
}

// Self-test of the panel kernel's bounded wait: one thread waits with
// wait_stamp for a stamp that nothing writes (a zeroed word, column 1), with a
// short limit, into the panel's own error word; out[0] = 1 if it gave up.
__global__ void stamp_expiry_selftest_kernel(const unsigned long long* word, unsigned long long limit_ns,
                                             int* err, int* out) {
    if (threadIdx.x != 0) return;
    out[0] = wait_stamp(word, 1u, err, limit_ns) == 0 ? 1 : 0;
}

// both substitutions for nrhs <= SOLVE_RHS.  *launched stays false when the
// kernel cannot be launched here (the caller then takes the blocked form)
template <int N>
int solve_few(const double* LU, long long lda, int n, double* B, long long ldb, int nrhs, void* words, int* err,
              cudaStream_t s, bool* launched) {
    constexpr int L = Limbs<N>::L;
    const int nb = (n + BASE - 1) / BASE, sms = device_sms();
    int kw = 16;
    while (16 / kw < nrhs) kw /= 2;
    const size_t smem = solve_smem<L>(nrhs), half = (size_t)nb * BASE * nrhs * (L + 2);
    unsigned long long* w = (unsigned long long*)words;
    if (cudaMemsetAsync(w, 0, 2 * half * sizeof *w, s) != cudaSuccess) return OZLU_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb < sms ? nb : sms);
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const size_t most = solve_smem<L>(SOLVE_RHS);
    raise_smem_limit((const void*)solve_kernel<N, true>, (int)most);
    raise_smem_limit((const void*)solve_kernel<N, false>, (int)most);
    if (cudaLaunchKernelEx(&cfg, solve_kernel<N, true>, LU, lda, n, B, ldb, nrhs, kw, w, err) != cudaSuccess) {
        cudaGetLastError();
        return OZLU_OK;
    }
    *launched = true;
    return cudaLaunchKernelEx(&cfg, solve_kernel<N, false>, LU, lda, n, B, ldb, nrhs, kw, w + half, err) == cudaSuccess
               ? OZLU_OK
               : OZLU_ERR_CUDA;
}

// Launch the cooperative base-block kernel; returns false when the slice of
// rows does not fit in shared memory (the caller then uses column kernels).
template <int N>
bool base_block_coop(double* A, long long lda, int n, int c0, int b, int* ipiv, int* info, void* scratch,
                     int min_rows, cudaStream_t s) {
    constexpr int L = Limbs<N>::L;
    const int sms = device_sms();
    // at least min_rows rows per block: a small panel takes a few SMs and
    // leaves the rest to concurrent work.  Fewer rows a block shorten the trailing
    // updates beside the chain, more leave fewer keys to read: QD n = 1000, 6.59 ms
    // with 6 rows, 6.61 with 8, 6.91 with 12, 7.40 with 16, 9.7 with 32.  The batched
    // driver runs instances side by side and asks for 32 (48 uneven TD systems from
    // CUDA graphs 21.3 ms, with 24 rows 22.2), single factorisations for 8.  A program
    // that factors on several handles at once is served less well by 8: milliseconds
    // per QD factorisation on 1, 2, 4 and 8 streams, n = 300 1.63, 0.85, 0.48, 0.39 (16
    // rows: 1.87, 0.96, 0.51, 0.30), n = 1000 6.2, 4.0, 3.9, 3.9 (7.1, 3.9, 2.7, 2.6).
    const int g_rows = (n - c0 + min_rows - 1) / min_rows;
    for (int per_sm = 1; per_sm <= 2; ++per_sm) {
        int G = sms * per_sm;
        if (G > COOP_MAXG) G = COOP_MAXG;
        if (G > g_rows) G = g_rows < 1 ? 1 : g_rows;
        const int rows = (n - c0 + G - 1) / G;
        const size_t smem = sizeof(MPF<L>) * (size_t)rows * (b + 1);
        if (rows > 256 || smem > 200 * 1024 / per_sm) continue;
        // rows per lane of warp 0: two keep its values in registers (n to 9728 at
        // one block per SM); more rows only meet narrow blocks
        const auto kernel = rows <= 64 ? base_block_coop_kernel<N, 2> : base_block_coop_kernel<N, 8>;
        raise_smem_limit((const void*)kernel, (int)(smem < 1024 ? 1024 : smem));
        int active = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&active, kernel, COOP_THREADS, smem);
        if (active * sms < G) continue;
        auto* sc = reinterpret_cast<CoopScratch<L>*>(scratch);
        // cooperative launch (all blocks co-resident), also valid under stream capture
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(G);
        cfg.blockDim = dim3(COOP_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, kernel, A, lda, n, c0, b, rows, ipiv, info, sc) !=
            cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return true;
    }
    return false;
}

struct Ctx {
    ozlu_handle* h;
    int nc, p;
    const ozlu_opts* opts;
    double* A;
    long long lda;
    int n;
    int* ipiv;
    LuScratch* sc;
    int rc = 0;
};

double* at(const Ctx& c, long long i, long long j) { return c.A + (i + j * c.lda) * c.nc; }

// widest base block for the cooperative panel kernel: the caller's choice,
// else PBASE (measured fastest on GB300 for n from 512 to 4096; a block
// whose rows do not fit in shared memory is split by the recursion)
int coop_width(const Ctx& c, int) {
    if (c.opts && c.opts->panel_width) return c.opts->panel_width < PBASE ? c.opts->panel_width : PBASE;
    return PBASE;
}

// r_top >= 0: the unit lower triangle's BASE x BASE diagonal blocks from row
// r_top on are already converted, block q in slot q
template <int N>
void trsm_rec(Ctx& c, long long r, int b, long long j0, int ncols, bool lower, long long r_top = -1) {
    if (c.rc || ncols <= 0) return;
    // (a power of two: the halving recursion then ends on the BASE blocks)
    if (lower && r_top < 0 && b > BASE && (b & (b - 1)) == 0 && b / BASE <= TRI_SLOTS) {
        // every leaf's triangle in one launch, ahead of the recursion
        c.h->phase(PH_TRSM);
        launch(tri_convert_kernel<N>, dim3((BASE * BASE + 255) / 256, b / BASE), 256, 0, c.h->stream, 
            at(c, r, r), c.lda, BASE, 1, c.sc);
        c.h->count(1);
        r_top = r;
    }
    if (b <= BASE) {
        c.h->phase(PH_TRSM);
        const int slot = (lower && r_top >= 0) ? (int)((r - r_top) / BASE) : -1;
        trsm_base<N>(at(c, r, r), c.lda, at(c, r, j0), c.lda, b, ncols, lower ? 1 : 0, c.sc, c.h->stream, slot);
        c.h->count(slot < 0 ? 2 : 1);
        return;
    }
    const int b1 = b / 2;
    if (lower) {
        trsm_rec<N>(c, r, b1, j0, ncols, true, r_top);
        c.rc = c.rc ? c.rc : gemm_device(c.h, N, c.p, b - b1, ncols, b1, -1, at(c, r + b1, r), c.lda,
                                         at(c, r, j0), c.lda, 1, at(c, r + b1, j0), c.lda, c.opts);
        trsm_rec<N>(c, r + b1, b - b1, j0, ncols, true, r_top);
    } else {
        trsm_rec<N>(c, r + b1, b - b1, j0, ncols, false);
        c.rc = c.rc ? c.rc : gemm_device(c.h, N, c.p, b1, ncols, b - b1, -1, at(c, r, r + b1), c.lda,
                                         at(c, r + b1, j0), c.lda, 1, at(c, r, j0), c.lda, c.opts);
        trsm_rec<N>(c, r, b1, j0, ncols, false);
    }
}

// factor the panel block with top-left (r, r), width b, rows [r, n); row
// interchanges are applied across the outer panel columns [p0, p1)
template <int N>
void panel_rec(Ctx& c, int r, int b, int p0, int p1) {
    if (c.rc) return;
    cudaStream_t s = c.h->stream;
    // up to coop_width columns in one cooperative kernel when its rows fit
    // in shared memory (else the block is split further)
    if (b <= coop_width(c, r)) {
        c.h->phase(PH_PANEL);
        if (base_block_coop<N>(c.A, c.lda, c.n, r, b, c.ipiv, &c.sc->info, c.h->coop_scratch,
                               c.h->coop_min_rows, s)) {
            c.h->count(1);
            if (p0 < r || r + b < p1) {
                c.h->phase(PH_OTHER);
                laswp2<N>(c.A, c.lda, p0, r, r + b, p1, r, r + b, c.ipiv, c.sc->plist, s);
                c.h->count(1 + (p0 < r) + (r + b < p1));
            }
            c.h->stats.panel_launches += 1;
            return;
        }
    }
    if (b <= BASE) {
        c.h->count(1 + b);
        c.h->stats.panel_launches += 1 + b;
        {
            const int rows = c.n - r;
            const int blocks = rows > PIV_THREADS * PIV_BLOCKS ? PIV_BLOCKS
                                                               : (rows + PIV_THREADS - 1) / PIV_THREADS;
            launch(pivot_kernel<N>, blocks, PIV_THREADS, 0, s, c.A, c.lda, c.n, r, p0, p1, c.ipiv, c.sc);
        }
        for (int col = r; col < r + b; ++col) {
            const int rows = c.n - col - 1;
            if (rows <= 0) break;
            int blocks = (rows + STEP_ROWS - 1) / STEP_ROWS;
            if (blocks > MAXPART) blocks = MAXPART;
            launch(column_step_kernel<N>, blocks, 128, 0, s, c.A, c.lda, c.n, col, r + b, p0, p1, c.ipiv,
                                                          c.sc);
        }
        return;
    }
    const int b1 = b / 2;
    panel_rec<N>(c, r, b1, p0, p1);
    trsm_rec<N>(c, r, b1, r + b1, b - b1, true);
    if (!c.rc && c.n - r - b1 > 0)
        c.rc = gemm_device(c.h, N, c.p, c.n - r - b1, b - b1, b1, -1, at(c, r + b1, r), c.lda,
                           at(c, r, r + b1), c.lda, 1, at(c, r + b1, r + b1), c.lda, c.opts);
    panel_rec<N>(c, r + b1, b - b1, p0, p1);
}

}  // namespace

template <int N>
int getrf_device(ozlu_handle* h, int p, int n, double* A, long long lda, int* ipiv, int nb,
                 LuScratch* sc, const ozlu_opts* opts) {
    Ctx c{h, N, p, opts, A, lda, n, ipiv, sc};
    cudaStream_t s = h->stream;
    for (int r0 = 0; r0 < n && !c.rc; r0 += nb) {
        const int b = nb < n - r0 ? nb : n - r0;
        panel_rec<N>(c, r0, b, r0, r0 + b);
        // (P2) interchanges on the columns left and right of the panel
        h->phase(PH_OTHER);
        h->count((r0 > 0) + (r0 + b < n));
        laswp2<N>(A, lda, 0, r0, r0 + b, n, r0, r0 + b, ipiv, sc->plist, s);
        if (r0 + b < n) {
            // (P3) U12 = L11^-1 A12
            trsm_rec<N>(c, r0, b, r0 + b, n - r0 - b, true);
            // (P4) A22 <- A22 - L21 U12
            if (!c.rc && opts && opts->native) {
                h->phase(PH_GEMM);
                const int mm = n - r0 - b;
                dim3 grid((mm + 15) / 16, (mm + 15) / 16);
                launch(naive_update_kernel<N>, grid, 256, 0, s, at(c, r0 + b, r0), lda, at(c, r0, r0 + b), lda,
                                                            at(c, r0 + b, r0 + b), lda, mm, mm, b);
                h->count(1);
            } else if (!c.rc) {
                c.rc = gemm_device(h, N, p, n - r0 - b, n - r0 - b, b, -1, at(c, r0 + b, r0), lda,
                                   at(c, r0, r0 + b), lda, 1, at(c, r0 + b, r0 + b), lda, opts);
            }
        }
    }
    h->phase(-1);
    if (!c.rc && cudaGetLastError() != cudaSuccess) c.rc = OZLU_ERR_CUDA;
    return c.rc;
}

template <int N>
int getrs_device(ozlu_handle* h, int p, int n, int nrhs, double* LU, long long lda, const int* ipiv,
                 double* B, long long ldb, const ozlu_opts* opts, LuScratch* sc) {
    cudaStream_t s = h->stream;
    // options that no plan of the updates meets are refused whichever form runs
    const int refused = n > BASE ? check_plan(h, p, BASE, opts) : OZLU_OK;
    if (refused) return refused;
    if (h->wait_limit)  // test hook: a wait that runs out, on a word that nothing writes
        stamp_expiry_selftest_kernel<<<1, 32, 0, s>>>((const unsigned long long*)(h->dev_err + 8), (unsigned long long)h->wait_limit,
                                                       h->dev_err, h->dev_err + 1);
    h->phase(PH_OTHER);
    laswp_all<N>(B, ldb, nrhs, n, ipiv, sc->plist, s);
    h->count(2 * ((n + LMAXB - 1) / LMAXB));
    int rc = 0;
    if (nrhs <= SOLVE_RHS) {
        constexpr int W = Limbs<N>::L + 2;
        const size_t rows = (size_t)(n + BASE - 1) / BASE * BASE;
        bool launched = false;
        rc = ensure_unmoved(h, h->solve_ws, 2 * sizeof(unsigned long long) * rows * nrhs * W);
        h->phase(PH_TRSM);
        if (!rc) rc = solve_few<N>(LU, lda, n, B, ldb, nrhs, h->solve_ws.base, h->dev_err, s, &launched);
        if (rc || launched) {
            h->count(2);
            h->phase(-1);
            return !rc && cudaGetLastError() != cudaSuccess ? OZLU_ERR_CUDA : rc;
        }
    }
    auto L = [&](long long i, long long j) { return LU + (i + j * lda) * N; };
    auto X = [&](long long i) { return B + i * N; };
    h->phase(PH_TRSM);
    h->count(4 * ((n + BASE - 1) / BASE));
    for (int r = 0; r < n && !rc; r += BASE) {
        const int b = BASE < n - r ? BASE : n - r;
        trsm_base<N>(L(r, r), lda, X(r), ldb, b, nrhs, 1, sc, s);
        if (r + b < n)
            rc = gemm_device(h, N, p, n - r - b, nrhs, b, -1, L(r + b, r), lda, X(r), ldb, 1,
                             X(r + b), ldb, opts);
    }
    const int last = ((n - 1) / BASE) * BASE;
    for (int r = last; r >= 0 && !rc; r -= BASE) {
        const int b = BASE < n - r ? BASE : n - r;
        trsm_base<N>(L(r, r), lda, X(r), ldb, b, nrhs, 0, sc, s);
        if (r > 0)
            rc = gemm_device(h, N, p, r, nrhs, b, -1, L(0, r), lda, X(r), ldb, 1, X(0), ldb, opts);
    }
    h->phase(-1);
    if (!rc && cudaGetLastError() != cudaSuccess) rc = OZLU_ERR_CUDA;
    return rc;
}

namespace {
size_t align256(size_t v) { return (v + 255) / 256 * 256; }
}  // namespace

int lu_scratch(ozlu_handle* h, LuScratch** out);
int coop_reset(ozlu_handle* h, int nc, int n, cudaStream_t s);

namespace {
// info of one factorisation: the first zero pivot (1-based), or
// -OZLU_ERR_TIMEOUT when a bounded wait of the panel kernel (its error word)
// or of a tensor-core GEMM (the handle's error word) gave up
__global__ void finish_kernel(int* info_out, const LuScratch* sc, const int* coop, const int* gerr) {
    int v = sc->info;
    if (coop[0]) v = -coop[0];
    else if (*gerr) v = -*gerr;
    *info_out = v;
}

}  // namespace

int launch_mbar_expiry_selftest(long long limit, int* err, int* out, cudaStream_t s);

// which = 1: the panel's stamp wait, then the factorisation's finish step
// (info); which = 2: the tensor-core GEMM's mbarrier wait.  out (host, 3
// ints): whether the wait gave up, the error word, info (which = 1).
int wait_expiry_selftest(ozlu_handle* h, int which, long long limit, int* out) {
    LuScratch* sc;
    int rc = lu_scratch(h, &sc);
    if (rc) return rc;
    cudaStream_t s = h->stream;
    int* gerr = err_word(h);
    if (!gerr) return OZLU_ERR_NOMEM;
    if (cudaMemsetAsync(sc, 0, sizeof(LuScratch), s)) return OZLU_ERR_CUDA;
    if ((rc = coop_reset(h, 4, 1, s))) return rc;
    if ((rc = clear_err_word(h))) return rc;
    // the candidate area of the scratch (zeroed above) holds a stamp word that
    // nothing writes and the kernel's flag
    unsigned long long* word = reinterpret_cast<unsigned long long*>(&sc->pval[0][0]);
    int* flag = &sc->pidx[0];
    if (which == 1) {
        stamp_expiry_selftest_kernel<<<1, 32, 0, s>>>(word, (unsigned long long)limit,
                                                       (int*)h->coop_scratch, flag);
        finish_kernel<<<1, 1, 0, s>>>(&sc->result, sc, (const int*)h->coop_scratch, gerr);
    } else if (which == 2) {
        if ((rc = launch_mbar_expiry_selftest(limit, gerr, flag, s))) return rc;
        finish_kernel<<<1, 1, 0, s>>>(&sc->result, sc, (const int*)h->coop_scratch, gerr);
    } else {
        return -2;
    }
    if (cudaGetLastError() != cudaSuccess) return OZLU_ERR_CUDA;
    int host[3] = {0, 0, 0};
    if (cudaMemcpyAsync(&host[0], flag, sizeof(int), cudaMemcpyDeviceToHost, s) ||
        cudaMemcpyAsync(&host[1], which == 1 ? (const int*)h->coop_scratch : gerr, sizeof(int),
                        cudaMemcpyDeviceToHost, s) ||
        cudaMemcpyAsync(&host[2], &sc->result, sizeof(int), cudaMemcpyDeviceToHost, s) ||
        cudaStreamSynchronize(s))
        return OZLU_ERR_CUDA;
    for (int i = 0; i < 3; ++i) out[i] = host[i];
    return host[2] < 0 ? -host[2] : OZLU_OK;
}

// one factorisation on device pointers (the batched driver calls it per
// instance on its own streams); info of the instance goes to *info_out
int getrf_one(ozlu_handle* h, int nc, int p, int n, double* A, long long lda, int* ipiv, int nb, int* info_out,
              const ozlu_opts* opts) {
    LuScratch* sc;
    int rc = lu_scratch(h, &sc);
    if (rc) return rc;
    cudaStream_t s = h->stream;
    // the unblocked naive comparison of Sec. 3.4: b = 1, every column's
    // rank-1 update of the whole trailing matrix in expansion arithmetic
    if (opts && opts->native == 2) nb = 1;
    if (cudaMemsetAsync(sc, 0, sizeof(LuScratch), s)) return OZLU_ERR_CUDA;
    if ((rc = coop_reset(h, nc, n, s))) return rc;
    if ((rc = clear_err_word(h))) return rc;
    if (n > 0) {
        switch (nc) {
            case 2: rc = getrf_device<2>(h, p, n, A, lda, ipiv, nb, sc, opts); break;
            case 3: rc = getrf_device<3>(h, p, n, A, lda, ipiv, nb, sc, opts); break;
            default: rc = getrf_device<4>(h, p, n, A, lda, ipiv, nb, sc, opts); break;
        }
    }
    if (rc) return rc;
    finish_kernel<<<1, 1, 0, s>>>(info_out, sc, (const int*)h->coop_scratch, h->dev_err);
    h->count(1);
    return cudaGetLastError() == cudaSuccess ? OZLU_OK : OZLU_ERR_CUDA;
}

int getrs_one(ozlu_handle* h, int nc, int p, int n, int nrhs, const double* LU, long long lda, const int* ipiv,
              double* B, long long ldb, const ozlu_opts* opts, bool clear) {
    LuScratch* sc;
    int rc = lu_scratch(h, &sc);
    if (rc) return rc;
    if (clear && (rc = clear_err_word(h))) return rc;
    switch (nc) {
        case 2: return getrs_device<2>(h, p, n, nrhs, (double*)LU, lda, ipiv, B, ldb, opts, sc);
        case 3: return getrs_device<3>(h, p, n, nrhs, (double*)LU, lda, ipiv, B, ldb, opts, sc);
        default: return getrs_device<4>(h, p, n, nrhs, (double*)LU, lda, ipiv, B, ldb, opts, sc);
    }
}

int lu_scratch(ozlu_handle* h, LuScratch** out) {
    if (!h->lu_scratch) {
        if (!dev_alloc(&h->lu_scratch, sizeof(LuScratch))) return OZLU_ERR_NOMEM;
    }
    if (!h->coop_scratch) {
        h->coop_bytes = std::max(std::max(sizeof(CoopScratch<Limbs<2>::L>), sizeof(CoopScratch<Limbs<3>::L>)),
                                 sizeof(CoopScratch<Limbs<4>::L>));
        if (!dev_alloc(&h->coop_scratch, h->coop_bytes)) {
            h->coop_scratch = nullptr;
            return OZLU_ERR_NOMEM;
        }
    }
    *out = (LuScratch*)h->lu_scratch;
    return OZLU_OK;
}

// the error word and the tagged words of the blocks a panel of n rows can have
// start at zero for every factorisation
int coop_reset(ozlu_handle* h, int nc, int n, cudaStream_t s) {
    int G = (n + h->coop_min_rows - 1) / h->coop_min_rows;
    if (G > 2 * device_sms()) G = 2 * device_sms();
    if (G > COOP_MAXG) G = COOP_MAXG;
    const dim3 grid(G < 1 ? 1 : G, COOP_DEPTH);
    // the slot layout is that of the panel kernel's limb count for nc
    constexpr int L2 = Limbs<2>::L, L3 = Limbs<3>::L, L4 = Limbs<4>::L;
    switch (nc) {
        case 2: coop_reset_kernel<L2><<<grid, 256, 0, s>>>((CoopScratch<L2>*)h->coop_scratch); break;
        case 3: coop_reset_kernel<L3><<<grid, 256, 0, s>>>((CoopScratch<L3>*)h->coop_scratch); break;
        default: coop_reset_kernel<L4><<<grid, 256, 0, s>>>((CoopScratch<L4>*)h->coop_scratch); break;
    }
    h->count(1);
    return cudaGetLastError() == cudaSuccess ? OZLU_OK : OZLU_ERR_CUDA;
}

// Panel width by measurement (nb = 0 in ozlu_getrf and the batched LU): the
// candidates 64, 128, 256 and 512 (not above n) each factor a scratch copy of
// A twice on the handle's stream, the second run timed with events (the first
// grows workspaces and lets the back-end autotuner see the new shapes); the
// fastest is cached per (nc, p, log2 n, back-end).  Never inside a capture.
int tune_nb(ozlu_handle* h, int nc, int p, int n, const double* A, long long lda, const ozlu_opts* opts,
            int* nb_out) {
    int lgn = 0;
    while ((1 << lgn) < n) ++lgn;
    const int be = opts ? opts->backend : 0;
    const auto key = std::make_tuple(nc, p, lgn, be);
    auto it = h->tuned_nb.find(key);
    if (it != h->tuned_nb.end()) {
        *nb_out = it->second;
        h->stats.tuned_nb = it->second;
        return OZLU_OK;
    }
    if (n <= 64 || h->capturing) {
        *nb_out = n <= 64 ? (n > 0 ? n : 1) : 256;
        return OZLU_OK;
    }
    ozlu_opts o;
    memset(&o, 0, sizeof o);
    if (opts) o = *opts;
    o.graph = 0;
    const size_t abytes = align256(sizeof(double) * nc * (size_t)n * n);
    int rc = h->nb_ws.ensure(abytes + align256(sizeof(int) * (size_t)n) + 256);
    if (rc) return rc;
    double* Ac = (double*)h->nb_ws.base;
    int* ipv = (int*)((char*)h->nb_ws.base + abytes);
    int* inf = (int*)((char*)ipv + align256(sizeof(int) * (size_t)n));
    cudaStream_t s = h->stream;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const bool timing = h->timing;
    h->timing = false;
    float best = 1e30f;
    int choice = 256 < n ? 256 : n;
    const int cands[4] = {64, 128, 256, 512};
    for (int c = 0; c < 4 && !rc; ++c) {
        const int nb = cands[c];
        if (nb > n && c > 0) break;
        for (int rep = 0; rep < 2 && !rc; ++rep) {
            if (cudaMemcpy2DAsync(Ac, sizeof(double) * nc * n, A, sizeof(double) * nc * lda, sizeof(double) * nc * n,
                                  n, cudaMemcpyDeviceToDevice, s) != cudaSuccess) {
                rc = OZLU_ERR_CUDA;
                break;
            }
            cudaEventRecord(e0, s);
            rc = getrf_one(h, nc, p, n, Ac, n, ipv, nb, inf, &o);
            cudaEventRecord(e1, s);
            if (rc) break;
            if (cudaEventSynchronize(e1) != cudaSuccess) { rc = OZLU_ERR_CUDA; break; }
            float ms = 0;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep == 1 && ms < best) { best = ms; choice = nb; }
        }
    }
    h->timing = timing;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    h->tuned_nb[key] = choice;
    h->stats.tuned_nb = choice;
    *nb_out = choice;
    return OZLU_OK;
}

// waits for the stream; OZLU_ERR_TIMEOUT if a bounded device wait gave up
int lu_result(ozlu_handle* h, cudaStream_t s, int* result) {
    LuScratch* sc = (LuScratch*)h->lu_scratch;
    if (cudaMemcpyAsync(result, &sc->result, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return OZLU_ERR_CUDA;
    return *result < 0 ? -*result : OZLU_OK;
}

}  // namespace ozlu

using namespace ozlu;

extern "C" int ozlu_getrf(ozlu_handle* h, int nc, int p, int n, double* A, long long lda, int* ipiv,
                          int nb, int* info, const ozlu_opts* opts) {
    if (!h) return -1;
    if (nc < 2 || nc > 4) return -2;
    if (p == 0) p = 53 * nc;
    if (p < 1 || p > 53 * nc) return -3;
    if (n < 0) return -4;
    if (!A && n) return -5;
    if (lda < (n > 1 ? n : 1)) return -6;
    if (!ipiv && n) return -7;
    if (nb < 0) return -8;
    if (!info) return -9;
    if (cudaSetDevice(h->device) != cudaSuccess) return OZLU_ERR_CUDA;
    cudaStream_t s = h->stream;
    LuScratch* sc;
    int rc = lu_scratch(h, &sc);
    if (rc) return rc;
    const bool dA = is_device_ptr(A), dP = is_device_ptr(ipiv), dI = is_device_ptr(info);
    if (opts && opts->graph && n > 0 && dA && dP && dI) {  // graph capture and replay
        if (nb == 0 && (rc = tune_nb(h, nc, p, n, A, lda, opts, &nb))) return rc;
        return ozlu_getrf_batched(h, nc, p, 1, &n, &A, &lda, &ipiv, info, nb, opts);
    }
    const size_t abytes = sizeof(double) * nc * (size_t)lda * (n ? n : 1);
    double* gA = A;
    int* gP = ipiv;
    if (!dA || !dP) {
        rc = h->stage.ensure(abytes + sizeof(int) * (size_t)(n + 1) + 512);
        if (rc) return rc;
        if (!dA) {
            gA = (double*)h->stage.base;
            if (cudaMemcpyAsync(gA, A, abytes, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA;
        }
        if (!dP) gP = (int*)((char*)h->stage.base + align256(abytes));
    }
    if (nb == 0 && n > 0 && (rc = tune_nb(h, nc, p, n, gA, lda, opts, &nb))) return rc;
    if (nb == 0) nb = 1;
    if ((rc = getrf_one(h, nc, p, n, gA, lda, gP, nb, &sc->result, opts))) return rc;
    int result = 0;
    if ((rc = lu_result(h, s, &result))) return rc;
    if (!dA && cudaMemcpyAsync(A, gA, abytes, cudaMemcpyDeviceToHost, s)) return OZLU_ERR_CUDA;
    if (n && gP != ipiv &&
        cudaMemcpyAsync(ipiv, gP, sizeof(int) * n, dP ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s))
        return OZLU_ERR_CUDA;
    if (cudaMemcpyAsync(info, &sc->info, sizeof(int), dI ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s))
        return OZLU_ERR_CUDA;
    if (!dA || !dP || !dI) return cuda_rc(cudaStreamSynchronize(s));
    return OZLU_OK;
}

extern "C" int ozlu_debug_wait_expiry(ozlu_handle* h, int which, long long limit, int* out) {
    if (!h) return -1;
    if (which != 1 && which != 2) return -2;
    if (limit < 1) return -3;
    if (!out) return -4;
    if (cudaSetDevice(h->device) != cudaSuccess) return OZLU_ERR_CUDA;
    return wait_expiry_selftest(h, which, limit, out);
}

extern "C" int ozlu_getrs(ozlu_handle* h, int nc, int p, int n, int nrhs, const double* LU,
                          long long lda, const int* ipiv, double* B, long long ldb,
                          const ozlu_opts* opts) {
    if (!h) return -1;
    if (nc < 2 || nc > 4) return -2;
    if (p == 0) p = 53 * nc;
    if (p < 1 || p > 53 * nc) return -3;
    if (n < 0) return -4;
    if (nrhs < 0) return -5;
    if (!LU && n) return -6;
    if (lda < (n > 1 ? n : 1)) return -7;
    if (!ipiv && n) return -8;
    if (!B && n && nrhs) return -9;
    if (ldb < (n > 1 ? n : 1)) return -10;
    if (n == 0 || nrhs == 0) return OZLU_OK;
    if (cudaSetDevice(h->device) != cudaSuccess) return OZLU_ERR_CUDA;
    cudaStream_t s = h->stream;
    LuScratch* sc;
    int rc0 = lu_scratch(h, &sc);
    if (rc0) return rc0;
    if ((rc0 = clear_err_word(h))) return rc0;
    const bool dL = is_device_ptr(LU), dP = is_device_ptr(ipiv), dB = is_device_ptr(B);
    if (opts && opts->graph && dL && dP && dB)  // graph capture and replay
        return ozlu_getrs_batched(h, nc, p, 1, &n, nrhs, &LU, &lda, &ipiv, &B, &ldb, opts);
    const size_t lbytes = sizeof(double) * nc * (size_t)lda * n;
    const size_t bbytes = sizeof(double) * nc * (size_t)ldb * nrhs;
    const double* gL = LU;
    const int* gP = ipiv;
    double* gB = B;
    int rc = 0;
    if (!dL || !dP || !dB) {
        rc = h->stage.ensure(align256(lbytes) + align256(bbytes) + sizeof(int) * (size_t)n + 256);
        if (rc) return rc;
        char* base = (char*)h->stage.base;
        if (!dL) { gL = (double*)base; if (cudaMemcpyAsync((void*)gL, LU, lbytes, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA; }
        if (!dB) { gB = (double*)(base + align256(lbytes)); if (cudaMemcpyAsync(gB, B, bbytes, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA; }
        if (!dP) {
            int* t = (int*)(base + align256(lbytes) + align256(bbytes));
            if (cudaMemcpyAsync(t, ipiv, sizeof(int) * n, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA;
            gP = t;
        }
    }
    switch (nc) {
        case 2: rc = getrs_device<2>(h, p, n, nrhs, (double*)gL, lda, gP, gB, ldb, opts, sc); break;
        case 3: rc = getrs_device<3>(h, p, n, nrhs, (double*)gL, lda, gP, gB, ldb, opts, sc); break;
        default: rc = getrs_device<4>(h, p, n, nrhs, (double*)gL, lda, gP, gB, ldb, opts, sc); break;
    }
    if (rc) return rc;
    if (!dB && cudaMemcpyAsync(B, gB, bbytes, cudaMemcpyDeviceToHost, s)) return OZLU_ERR_CUDA;
    if (!dL || !dP || !dB) return finish_call(h);
    return OZLU_OK;
}
