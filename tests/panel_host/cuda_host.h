// A thread block on the CPU, for tests of kernels whose warps work side by side:
// every CUDA thread is a coroutine of one operating-system thread (blocks run in
// threads of their own), warp-wide operations and barriers are rendezvous, and
// the order in which the warps go on is the caller's, so that a warp can be held
// back for as long as the kernel's own synchronisation allows.
#pragma once

#include <sched.h>
#include <sys/mman.h>
#include <ucontext.h>

#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <random>
#include <vector>

#define __device__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __shared__ thread_local
#define __align__(n) __attribute__((aligned(n)))
#define __launch_bounds__(...)

static inline int __clz(uint32_t x) { return x ? __builtin_clz(x) : 32; }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline long long __double_as_longlong(double d) { long long r; memcpy(&r, &d, 8); return r; }
static inline double __longlong_as_double(long long x) { double r; memcpy(&r, &x, 8); return r; }
static inline uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static inline float __frcp_rn(float x) { volatile float one = 1.0f; return one / x; }
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) {
    s &= 31;
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
static inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) {
    s &= 31;
    return s ? (lo >> s) | (hi << (32 - s)) : lo;
}
static inline int min(int a, int b) { return a < b ? a : b; }
static inline int max(int a, int b) { return a > b ? a : b; }
static inline int atomicExch(int* p, int v) { return __atomic_exchange_n(p, v, __ATOMIC_RELAXED); }

struct Dim { unsigned x = 0, y = 0, z = 0; };
static thread_local Dim threadIdx, blockIdx, blockDim, gridDim;

namespace host {

constexpr size_t STACK = 256 * 1024;

struct Thread {
    ucontext_t ctx;
    int tid = 0;
    bool waits = false, done = false;
    const void* seen[64] = {nullptr};  // words read last, to tell a poll that found nothing new
    uint64_t val[64] = {0};
};

struct Warp {
    uint64_t word[2][32] = {{0}};
    int arrived = 0, gen = 0;
    bool parked = false;  // its last poll found nothing new
};

struct Barrier {
    int count = 0;
    std::vector<int> waiting;
};

// order(warps) -> the warp to go on with, of those that can
using Order = std::function<int(const std::vector<int>&)>;

struct Block {
    std::vector<Thread> t;
    std::vector<Warp> w;
    Barrier bar[16];
    ucontext_t sched;
    std::function<void()> body;
    int cur = 0;

    void leave() {  // to the scheduler and back
        const int me = cur;
        swapcontext(&t[me].ctx, &sched);
        threadIdx.x = (unsigned)me;
    }
    static void entry();
    void run(int threads, const std::function<void()>& kernel, const Order& order);
};

static thread_local Block* block;

inline void Block::entry() {
    Block* b = block;
    threadIdx.x = (unsigned)b->cur;
    b->body();
    b->t[b->cur].done = true;
    b->leave();
}

inline void Block::run(int threads, const std::function<void()>& kernel, const Order& order) {
    block = this;
    body = kernel;
    t = std::vector<Thread>(threads);
    w = std::vector<Warp>(threads / 32);
    char* mem = (char*)mmap(nullptr, STACK * threads, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (mem == (char*)MAP_FAILED) abort();
    for (int i = 0; i < threads; ++i) {
        t[i].tid = i;
        getcontext(&t[i].ctx);
        t[i].ctx.uc_stack.ss_sp = mem + STACK * i;
        t[i].ctx.uc_stack.ss_size = STACK;
        t[i].ctx.uc_link = &sched;
        makecontext(&t[i].ctx, (void (*)())&Block::entry, 0);
    }
    long long idle = 0;
    std::vector<int> can;
    for (;;) {
        can.clear();
        bool live = false, parked = false;
        for (int k = 0; k < (int)w.size(); ++k) {
            bool runs = false;
            for (int i = 32 * k; i < 32 * k + 32; ++i) {
                live |= !t[i].done;
                runs |= !t[i].done && !t[i].waits;
            }
            if (runs && !w[k].parked) can.push_back(k);
            parked |= runs && w[k].parked;
        }
        if (!live) break;
        if (can.empty()) {
            if (!parked || ++idle > 20000000) { fprintf(stderr, "no warp can go on\n"); abort(); }
            for (auto& x : w) x.parked = false;
            if (gridDim.x > 1) sched_yield();
            continue;
        }
        const int k = order(can);
        // one round of the warp: each of its threads up to its next wait or poll
        for (int i = 32 * k; i < 32 * k + 32; ++i)
            if (!t[i].done && !t[i].waits) {
                cur = i;
                swapcontext(&sched, &t[i].ctx);
            }
    }
    munmap(mem, STACK * threads);
}

// every lane's word to every lane of the warp
inline const uint64_t* exchange(uint64_t v) {
    Block& b = *block;
    const int me = b.cur, k = me / 32;
    Warp& w = b.w[k];
    const int g = w.gen & 1;
    w.word[g][me % 32] = v;
    if (++w.arrived == 32) {
        w.arrived = 0;
        ++w.gen;
        for (int i = 32 * k; i < 32 * k + 32; ++i) b.t[i].waits = false;
    } else {
        b.t[me].waits = true;
        b.leave();
    }
    return w.word[g];
}

inline void barrier(int id, int threads, bool wait) {
    Block& b = *block;
    const int me = b.cur;
    Barrier& s = b.bar[id];
    if (++s.count == threads) {
        s.count = 0;
        for (int i : s.waiting) b.t[i].waits = false;
        s.waiting.clear();
    } else if (wait) {
        s.waiting.push_back(me);
        b.t[me].waits = true;
        b.leave();
    }
}

template <typename T> inline uint64_t bits(T v) { uint64_t r = 0; memcpy(&r, &v, sizeof v); return r; }
template <typename T> inline T from(uint64_t r) { T v; memcpy(&v, &r, sizeof v); return v; }

}  // namespace host

template <typename T> static inline T __shfl_sync(unsigned, T v, int src) {
    return host::from<T>(host::exchange(host::bits(v))[src & 31]);
}
template <typename T> static inline T __shfl_xor_sync(unsigned, T v, int o) {
    const int lane = host::block->cur & 31;
    return host::from<T>(host::exchange(host::bits(v))[lane ^ o]);
}
static inline unsigned __ballot_sync(unsigned, bool p) {
    const uint64_t* w = host::exchange(p);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r |= (unsigned)w[i] << i;
    return r;
}
static inline bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
static inline bool __all_sync(unsigned m, bool p) { return __ballot_sync(m, p) == 0xffffffffu; }
static inline unsigned __reduce_max_sync(unsigned, unsigned v) {
    const uint64_t* w = host::exchange(v);
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r = w[i] > r ? (unsigned)w[i] : r;
    return r;
}
static inline unsigned __reduce_min_sync(unsigned, unsigned v) {
    const uint64_t* w = host::exchange(v);
    unsigned r = 0xffffffffu;
    for (int i = 0; i < 32; ++i) r = w[i] < r ? (unsigned)w[i] : r;
    return r;
}
static inline int __reduce_add_sync(unsigned, int v) {
    const uint64_t* w = host::exchange((uint32_t)v);
    int r = 0;
    for (int i = 0; i < 32; ++i) r += (int)w[i];
    return r;
}
static inline void __syncwarp() { host::exchange(0); }
static inline void __syncthreads() { host::barrier(0, (int)host::block->t.size(), true); }

namespace ozlu {
// the accesses that device code makes in inline assembly
static inline unsigned long long global_ns() { return 0; }  // (a wait never expires; the scheduler finds a deadlock)
static inline unsigned long long ld_relaxed(const unsigned long long* p) {
    const unsigned long long v = __atomic_load_n(p, __ATOMIC_ACQUIRE);
    host::Block& b = *host::block;
    host::Thread& t = b.t[b.cur];
    const int h = (int)(((uintptr_t)p >> 3) % 61);
    if (t.seen[h] == p && t.val[h] == v) {
        b.w[b.cur / 32].parked = true;
        b.leave();
    }
    t.seen[h] = p;
    t.val[h] = v;
    return v;
}
static inline void st_relaxed(unsigned long long* p, unsigned long long v) { __atomic_store_n(p, v, __ATOMIC_RELEASE); }
static inline void bar_sync(int id, int threads) {
    __syncwarp();
    host::barrier(id, threads, true);
}
static inline void bar_arrive(int id, int threads) {
    __syncwarp();
    host::barrier(id, threads, false);
}
}  // namespace ozlu
