// (S4) residue GEMMs on the fifth-generation tensor cores of sm_103a, with
// the (S5) modular epilogue.
//
// Back-ends (Sec. 4.2.3):
//   FP8  E4M3, balanced base-17 digits of each centered residue, Eq. (15):
//        r = 17 d1 + d0, |d0| <= 8, |d1| <= 7, |d0 + d1| <= 15.  Three digit
//        planes per residue (d0, d1, d0 + d1) and three fp32 accumulators
//        P00, P11, Pss give the exact product by Karatsuba,
//        r r' summed = P00 + 17 (Pss - P00 - P11) + 289 P11.
//   FP16 the centered residue itself (|r| <= 127 is exact in binary16), one
//        plane, one fp32 accumulator; exact while K_pad S 127^2 < 2^24
//        (Eq. (14)).
//   INT8 the same planes at any K: an accumulator takes 1024 products of
//        residues, and the epilogue folds the accumulators of a product into
//        each other modulo m (MULTI).  QD, 1024^3: 241 us; the FP8 plan's three
//        planes take 342.
// Both rely on the fp32 tensor-core accumulation being exact for integer
// sums below 2^24; the parity tests check it bit for bit.
//
// Kernel: persistent, one CTA per SM over 128 x 128 output tiles.  A unit is one
// tile of a triple of moduli (packed results) or of one modulus (bytes); its
// plane products follow one another through a ring of four accumulators in
// TMEM (4 x 128 columns), so the MMAs of the next products run while the
// epilogue reduces the last.
//   warp 0: TMA producer (cp.async.bulk.tensor, SWIZZLE_128B, no multicast)
//   warp 1: one thread issues tcgen05.mma (M = 128, N = 128, K = 32 bytes
//           per instruction) into TMEM, tcgen05.commit frees smem stages and
//           hands a finished accumulator to the epilogue
//   warps 2-17: epilogue (four warps per TMEM lane quarter, each on a quarter
//           of the columns), tcgen05.ld 32x32b, frees the accumulator at once,
//           then t_l = (C y_l) mod m_l.
// The kernel is bound by shared memory: every operand byte is written once by
// TMA and read once by the 128 x 128 MMAs (about 530 cycles a stage where the
// MMAs alone need 256), with the epilogue close behind at K = 256.  The
// reduction therefore runs on the binary32 pipe (eight full-rate instructions
// per value, all exact: fma with the rounding constant 1.5 2^23 for the first
// quotient, fma rounding down for the floor of the second), where integer
// code with its float conversions took about 40, and a triple's three t values
// leave as the one 32-bit word u_q (CrtTab) that the CRT needs, a 128-byte
// store a warp instead of three of 32 bytes.
// FP16, QD, 3840 x 3840 x 256: 891 us (1928 before); FP8, QD, 1024^3: 342 us (534
// before).  Clusters of two CTAs that share the B tile by multicast (a quarter
// less L2 traffic) measured the same, 893 us.
// Every mbarrier wait has an iteration limit; on expiry the CTA records
// OZLU_ERR_TIMEOUT, stops issuing work, and releases its TMEM.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "launch.cuh"
#include "ozlu_internal.h"
#include "tables.h"

namespace ozlu {
namespace {

constexpr int BM = 128, BN = 128, BK = 128;  // BK in bytes: one 128-byte swizzle row
constexpr int STAGES = 6;
constexpr int THREADS = 576;          // producer, MMA and 16 epilogue warps
constexpr int EPI = THREADS - 64;     // epilogue threads
constexpr int NBUF = 4;               // accumulators in TMEM
constexpr int TILE = BM * BK;                // 16 KiB per operand stage
constexpr long long WAIT_LIMIT = 1ll << 24;  // iterations of ~100 ns

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// one lane of a converged warp.  The warp's control flow stays uniform (loop
// state and descriptors in uniform registers); a loop inside `if (lane == 0)`
// took about 700 cycles to issue a stage of four MMAs.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r != 0;
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(b)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(b)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait: false (and the error word set) after `limit` tries
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* err, volatile int* abort,
                                          long long limit = WAIT_LIMIT) {
    if (mbar_try_wait(b, parity)) return true;
    long long it = 0;
    while (!mbar_try_wait(b, parity)) {
        if (*abort) return false;
        if (++it > limit) {
            atomicExch(err, OZLU_ERR_TIMEOUT);
            *abort = 1;
            return false;
        }
        // the ring's waits are short: sleeping at once would add to each of them
        if (it > 32) __nanosleep(64);
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::
            "r"(su32(dst)),
        "l"(tm), "r"(x), "r"(y), "r"(su32(bar))
        : "memory");
}

// shared-memory matrix descriptor: K-major, SWIZZLE_128B, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
    const uint64_t addr = su32(p);
    return ((addr & 0x3ffff) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

template <bool FP8>
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    if (FP8)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
    else
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(su32(b))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// 1.5 2^23: adding it rounds a binary32 value below 2^22 to an integer, whose
// low bits are then the low bits of the sum
constexpr float RINT = 12582912.0f;

// c mod m up to a multiple of m: |result| <= 0.54 m + 1, exact for |c| < 2^24
__device__ __forceinline__ float fold(float c, float m, float inv) {
    const float q = __fadd_rn(__fmaf_rn(c, inv, RINT), -RINT);
    return __fmaf_rn(-q, m, c);
}

// bits of RINT + (v mod m) for an integer 0 <= v < 2^17, invu the float above
// 1 / m: v invu exceeds v / m by less than 1 / 255, so its floor is exact
__device__ __forceinline__ uint32_t floor_mod_bits(float v, float m, float invu) {
    const float k = __fadd_rn(__fmaf_rd(v, invu, RINT), -RINT);
    return __float_as_uint(__fadd_rn(__fmaf_rn(-k, m, v), RINT));
}

// The CTAs walk the units (gi, q, tm, tn) with stride gridDim.x, tn fastest, so
// those in flight share A row panels and B column panels in L2.
template <bool FP8, bool PACK, bool MULTI>
__global__ void __launch_bounds__(THREADS, 1) gemm_tc05_kernel(
    const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int m, int n,
    int Mpad, int Npad, int KB, int chunk, const __grid_constant__ GemmTab tab, void* T,
    int* err) {
    constexpr int P = FP8 ? 3 : 1;                // planes (products per modulus)
    constexpr int LG = PACK ? 3 : 1;              // moduli per unit
    // columns of an accumulator read at a time: 32 words more would not fit in
    // the 96 registers a thread beside the packed ones
    constexpr int LD = PACK && (FP8 || MULTI) ? 16 : 32;
    constexpr uint32_t TMEM_COLS = NBUF * BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sa = sm;
    uint8_t* sb = sm + STAGES * TILE;
    uint64_t* full = (uint64_t*)(sm + 2 * STAGES * TILE);
    uint64_t* empty = full + STAGES;
    uint64_t* accf = empty + STAGES;   // [NBUF] accumulator ready (MMA -> epilogue)
    uint64_t* acce = accf + NBUF;      // [NBUF] accumulator free (epilogue -> MMA)
    uint32_t* tmem_slot = (uint32_t*)(acce + NBUF);
    volatile int* abort = (volatile int*)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int TM = Mpad / BM, TN = Npad / BN;
    const int NQ = PACK ? tab.NT : tab.N;
    const int units = TM * TN * NQ * tab.G;
    const int S = tab.S;
    // unit -> (tm, tn, q, gi), its moduli [q LG, l1) and items per product
    // (pair terms x K blocks)
    auto decode = [&](int t, int& tm, int& tn, int& q, int& gi, int& l1, int& ta0, int& items) {
        tn = t % TN;
        int r = t / TN;
        tm = r % TM;
        r /= TM;
        q = r % NQ;
        gi = r / NQ;
        l1 = min(tab.N, q * LG + LG);
        const int g = tab.g0 + gi;
        ta0 = max(0, g - (S - 1));
        const int ta1 = min(g, S - 1);
        items = (ta1 - ta0 + 1) * KB;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < NBUF; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], EPI);
        }
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(tmem_slot)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = *tmem_slot;
    chain_enter();  // (the set-up above runs beside the conversion)

    if (warp == 0) {
        // position in the smem ring: stage s, parity of its pass; `issued`
        // (at most STAGES) stages hold copies that nobody may have waited for
        int s = 0, issued = 0;
        uint32_t par = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < units && ok; t += gridDim.x) {
            int tm, tn, q, gi, l1, ta0, items;
            decode(t, tm, tn, q, gi, l1, ta0, items);
            const int g = tab.g0 + gi, ta1 = min(g, S - 1);
            for (int l = q * LG; l < l1 && ok; ++l)
                for (int p = 0; p < P && ok; ++p)
                    for (int ta = ta0; ta <= ta1 && ok; ++ta) {
                        const int ya = ((l * S + ta) * P + p) * Mpad + tm * BM;
                        const int yb = ((l * S + g - ta) * P + p) * Npad + tn * BN;
                        for (int kb = 0, x = 0; kb < KB; ++kb, x += FP8 ? BK : BK / 2) {
                            if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], par ^ 1, err, abort))) { ok = false; break; }
                            if (elect_one()) {
                                mbar_expect_tx(&full[s], 2 * TILE);
                                tma_load_2d(sa + s * TILE, &tmA, x, ya, &full[s]);
                                tma_load_2d(sb + s * TILE, &tmB, x, yb, &full[s]);
                            }
                            __syncwarp();
                            issued = min(issued + 1, STAGES);
                            if (++s == STAGES) { s = 0; par ^= 1; }
                        }
                    }
        }
        if (!ok || *abort) {
            // let the copies already issued land before the CTA exits (bounded)
            for (; issued > 0; --issued) {
                if (--s < 0) { s = STAGES - 1; par ^= 1; }
                long long w = 0;
                while (!mbar_try_wait(&full[s], par) && ++w < WAIT_LIMIT) __nanosleep(64);
            }
        }
    } else if (warp == 1) {
        // kind::f8f6f4 E4M3 x E4M3 or kind::f16 F16 x F16 (format code 0 in both),
        // fp32 accumulate, K-major A and B, N = 128, M = 128
        const uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        const uint64_t da = smem_desc(sa), db = smem_desc(sb);
        // ring positions: smem stage s, accumulator b, with their parities
        int s = 0, b = 0;
        uint32_t par = 0, bpar = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < units && ok; t += gridDim.x) {
            int tm, tn, q, gi, l1, ta0, items;
            decode(t, tm, tn, q, gi, l1, ta0, items);
            const int prods = (l1 - q * LG) * P;
            for (int pd = 0, i1 = 0; pd < prods && ok; pd += MULTI ? i1 == items : 1) {
                // one accumulator: the next `chunk` K blocks of product pd
                const int i0 = !MULTI || i1 == items ? 0 : i1;
                i1 = MULTI ? min(items, i0 + chunk) : items;
                if (!__all_sync(0xffffffffu, mbar_wait(&acce[b], bpar ^ 1, err, abort))) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint32_t acc = tmem + (uint32_t)(b * BN);
                for (int i = i0; i < i1; ++i) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&full[s], par, err, abort))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;\n");
                    const uint64_t ad = da + (uint64_t)(s * (TILE >> 4)), bd = db + (uint64_t)(s * (TILE >> 4));
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < BK / 32; ++k)
                            mma<FP8>(acc, ad + 2 * k, bd + 2 * k, idesc, (i == i0 && k == 0) ? 0u : 1u);
                        mma_commit(&empty[s]);
                        if (i == i1 - 1) mma_commit(&accf[b]);
                    }
                    __syncwarp();
                    if (++s == STAGES) { s = 0; par ^= 1; }
                }
                if (++b == NBUF) { b = 0; bpar ^= 1; }
            }
        }
    } else {
        // epilogue warps: TMEM lane quarter = warp % 4; the k-th group of four
        // warps (from warp 2) takes the k-th quarter of the tile's columns
        const int lq = warp & 3;
        const int c0 = ((warp - 2) >> 2) * 32;
        const uint32_t lane_addr = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)c0;
        int b = 0;
        uint32_t bpar = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < units && ok; t += gridDim.x) {
            int tm, tn, q, gi, l1, ta0, items;
            decode(t, tm, tn, q, gi, l1, ta0, items);
            const int i = tm * BM + lq * 32 + lane;
            const int cols = min(32, n - tn * BN - c0);  // of this warp, may be <= 0
            uint32_t u[PACK ? 32 : 1];
            if (PACK) {
#pragma unroll
                for (int jj = 0; jj < 32; ++jj) u[PACK ? jj : 0] = tab.ucorr[q];
            }
            for (int l = q * LG; l < l1 && ok; ++l) {
                const GemmMod& M = tab.mod[l];
                const float md = M.m, inv = M.inv;
                float v[32];
                if (MULTI) {
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) v[jj] = 0.0f;
                }
                // (FP8: the planes; FP16: the accumulators of the one product)
                const int accs = FP8 ? P : (MULTI ? (items + chunk - 1) / chunk : 1);
#pragma unroll(FP8 ? 3 : 1)
                for (int p = 0; p < accs; ++p) {
                    // (the vote keeps the warp together for the loads that follow)
                    if (!ok || !__all_sync(0xffffffffu, mbar_wait(&accf[b], bpar, err, abort))) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;\n");
                    const float yp = M.y[p], off = M.off;
#pragma unroll
                    for (int h = 0; h < 32; h += LD) {
                        uint32_t r[LD];
                        tmem_ld(lane_addr + (uint32_t)(b * BN + h), r);
                        if (h + LD == 32) {
                            // the accumulator is in registers: the MMA warp may overwrite it
                            asm volatile("tcgen05.fence::before_thread_sync;\n");
                            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(su32(&acce[b])) : "memory");
                        }
#pragma unroll
                        for (int jj = 0; jj < LD; ++jj) {
                            const float c = __uint_as_float(r[jj]);
                            float& w = v[h + jj];
                            if (MULTI) w = fold(c + w, md, inv);
                            else w = __fmaf_rn(fold(c, md, inv), yp, p == 0 ? off : w);
                        }
                    }
                    if (++b == NBUF) { b = 0; bpar ^= 1; }
                }
                if (!ok) break;
                if (MULTI) {
                    const float yp = M.y[0], off = M.off;
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) v[jj] = __fmaf_rn(v[jj], yp, off);
                }
                const float invu = M.invu;
                if (PACK) {
                    const uint32_t cf = M.coef;
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) u[PACK ? jj : 0] += floor_mod_bits(v[jj], md, invu) * cf;
                } else if (i < m) {
                    uint8_t* out = (uint8_t*)T + ((size_t)gi * tab.N + l) * (size_t)m * n +
                                   (size_t)(tn * BN + c0) * m + i;
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj)
                        if (jj < cols) out[(size_t)jj * m] = (uint8_t)floor_mod_bits(v[jj], md, invu);
                }
            }
            if (PACK && ok && i < m) {
                uint32_t* out = (uint32_t*)T + ((size_t)gi * tab.NT + q) * (size_t)m * n +
                                (size_t)(tn * BN + c0) * m + i;
#pragma unroll
                for (int jj = 0; jj < 32; ++jj)
                    if (jj < cols) out[(size_t)jj * m] = u[PACK ? jj : 0];
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
    }
}

// Self-test of the bounded mbarrier wait: one thread waits with the kernel's
// own wait routine on a barrier nothing ever arrives at (phase 0 of a fresh
// barrier), with a short iteration limit; out[0] = 1 if the wait gave up.
// No TMA, MMA or TMEM is involved.
__global__ void mbar_expiry_selftest_kernel(long long limit, int* err, int* out) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    const bool ok = mbar_wait(&bar, 0, err, &abort_flag, limit);
    out[0] = ok ? 0 : 1;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

// 2-D map over a plane stack: inner dimension = Kpad elements, outer = rows
bool make_map(CUtensorMap* tm, const void* base, bool fp8, int Kpad, long long rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    const int esz = fp8 ? 1 : 2;
    cuuint64_t dims[2] = {(cuuint64_t)Kpad, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)Kpad * esz};
    cuuint32_t box[2] = {(cuuint32_t)(BK / esz), (cuuint32_t)BM};
    cuuint32_t estr[2] = {1, 1};
    return fn(tm, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (void*)base, dims,
              strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int launch_mbar_expiry_selftest(long long limit, int* err, int* out, cudaStream_t s) {
    mbar_expiry_selftest_kernel<<<1, 32, 0, s>>>(limit, err, out);
    return cudaGetLastError() == cudaSuccess ? OZLU_OK : OZLU_ERR_CUDA;
}

size_t tc05_smem_bytes() { return 2 * STAGES * TILE + 2 * STAGES * 8 + 2 * NBUF * 8 + 16 + 1024; }

// Packed results where every SM still gets four units or more; below that the
// coarser units (three moduli) leave SMs idle in the last round, and bytes (a
// unit per modulus) are taken.
bool tc05_packs(const GemmTab& tab, int Mpad, int Npad) {
    return (long long)(Mpad / BM) * (Npad / BN) * tab.NT * tab.G >= 4ll * device_sms();
}

int launch_gemm_tc05(bool fp8, bool pack, const void* RA, const void* RB, int m, int n, int Mpad, int Npad, int Kpad,
                     const GemmTab& tab, void* T, int* err, cudaStream_t s) {
    const int P = fp8 ? 3 : 1;
    CUtensorMap ta, tb;
    if (!make_map(&ta, RA, fp8, Kpad, (long long)tab.N * tab.S * P * Mpad)) return OZLU_ERR_UNSUPPORTED;
    if (!make_map(&tb, RB, fp8, Kpad, (long long)tab.N * tab.S * P * Npad)) return OZLU_ERR_UNSUPPORTED;
    const int KB = Kpad * (fp8 ? 1 : 2) / BK;
    // FP16: residues up to 127, so that 1024 products of two (16 K blocks) and
    // the folded rest of the accumulator before stay below 2^24 in binary32
    const int chunk = fp8 ? KB * tab.S : 1024 / (BK / 2);
    const size_t smem = tc05_smem_bytes();
    const int sms = device_sms();
    const long long units = (long long)(Mpad / BM) * (Npad / BN) * (pack ? tab.NT : tab.N) * tab.G;
    dim3 grid((unsigned)(units < sms ? units : sms));
    auto go = [&](auto kernel) {
        raise_smem_limit((const void*)kernel, (int)smem);
        launch(kernel, grid, THREADS, smem, s, ta, tb, m, n, Mpad, Npad, KB, chunk, tab, T, err);
    };
    if (fp8) pack ? go(gemm_tc05_kernel<true, true, false>) : go(gemm_tc05_kernel<true, false, false>);
    else if (KB * tab.S > chunk) pack ? go(gemm_tc05_kernel<false, true, true>) : go(gemm_tc05_kernel<false, false, true>);
    else pack ? go(gemm_tc05_kernel<false, true, false>) : go(gemm_tc05_kernel<false, false, false>);
    return cudaGetLastError() == cudaSuccess ? OZLU_OK : OZLU_ERR_CUDA;
}

}  // namespace ozlu
