// The panel kernel of the LU (csrc/panel.cuh) on the CPU, once for every order of
// its warps that the arguments name.
//
//   panel_host N n b rows order seed
//
// N components, n rows, b columns, `rows` rows a block; order "even" lets the warps
// go on in turn, "late" holds one warp after another back as long as possible
// (the seed says which order of preference), "mixed" draws a new preference every
// few steps; "plain" is no run of the kernel but the same factorisation as a plain
// loop, one element after another.  Prints the interchanges, info and the factored panel's words.
#include "cuda_host.h"

#include <algorithm>
#include <memory>
#include <numeric>
#include <string>
#include <thread>

#include "panel.cuh"

namespace ozlu {
namespace {
thread_local unsigned char smraw[1 << 20] __attribute__((aligned(16)));
}
}  // namespace ozlu

using namespace ozlu;

static host::Order make_order(const std::string& kind, uint64_t seed, int warps) {
    auto g = std::make_shared<std::mt19937_64>(seed);
    auto rank = std::make_shared<std::vector<int>>(warps);  // lower goes first
    std::iota(rank->begin(), rank->end(), 0);
    if (kind != "even") std::shuffle(rank->begin(), rank->end(), *g);
    auto left = std::make_shared<int>(0);
    if (kind == "even")
        return [left](const std::vector<int>& can) { return can[(size_t)(*left)++ % can.size()]; };
    return [=](const std::vector<int>& can) {
        if (kind == "mixed" && --*left < 0) {
            *left = (int)((*g)() % 300);
            std::shuffle(rank->begin(), rank->end(), *g);
        }
        return *std::min_element(can.begin(), can.end(), [&](int a, int b) { return (*rank)[a] < (*rank)[b]; });
    };
}

// columns in turn: the pivot (lowest row on ties), the multipliers x (1 / p), every
// other element y - l u; each operation rounded to L words
template <int N>
static void plain(double* A, int n, int b, int* ipiv, int* info) {
    constexpr int L = Limbs<N>::L;
    std::vector<MPF<L>> a((size_t)n * b);
    for (size_t e = 0; e < a.size(); ++e) a[e] = mpf_from_exp<L, N>(A + e * N);
    auto at = [&](int i, int j) -> MPF<L>& { return a[(size_t)j * n + i]; };
    for (int c = 0; c < b; ++c) {
        int p = c;
        for (int i = c + 1; i < n; ++i)
            if (mpf_abs_cmp<L>(at(i, c), at(p, c)) > 0) p = i;
        ipiv[c] = p + 1;
        if (mpf_zero<L>(at(p, c))) {
            if (*info == 0) *info = c + 1;
            continue;
        }
        for (int k = 0; k < b; ++k) std::swap(at(c, k), at(p, k));
        const MPF<L> r = mpf_recip<L>(at(c, c));
        for (int i = c + 1; i < n; ++i) {
            at(i, c) = mpf_mul<L>(at(i, c), r);
            for (int k = c + 1; k < b; ++k) at(i, k) = mpf_fms<L>(at(i, k), at(i, c), at(c, k));
        }
    }
    for (size_t e = 0; e < a.size(); ++e) mpf_to_exp<L, N>(a[e], A + e * N);
}

template <int N>
static void go(int n, int b, int rows, const std::string& order, uint64_t seed) {
    constexpr int L = Limbs<N>::L;
    std::vector<double> A((size_t)n * b * N, 0.0);
    std::mt19937_64 g(7);  // the same matrix for every order
    for (size_t e = 0; e < (size_t)n * b; ++e) {
        double x = std::ldexp((double)(g() >> 11), -53) * 2 - 1;
        for (int c = 0; c < N; ++c) {
            A[e * N + c] = x;
            x = std::ldexp(x * 0.7, -54);
        }
    }
    // rows and entries that make candidates zero or a power of two (no reciprocal to wait for)
    for (int j = 0; j < b; ++j)
        for (int i = 0; i < n; ++i)
            if (j % 16 == 5 || i % 11 == 3)
                for (int c = 0; c < N; ++c) A[((size_t)j * n + i) * N + c] = c ? 0.0 : (double)((int)(g() % 5) - 2);
    const int G = (n + rows - 1) / rows;
    std::vector<int> ipiv(b, 0);
    int info = 0;
    auto* sc = new CoopScratch<L>();
    memset((void*)sc, 0, sizeof *sc);
    std::vector<std::thread> blocks;
    if (order == "plain") plain<N>(A.data(), n, b, ipiv.data(), &info);
    for (int k = 0; k < G && order != "plain"; ++k)
        blocks.emplace_back([&, k] {
            blockIdx.x = (unsigned)k;
            gridDim.x = (unsigned)G;
            blockDim.x = COOP_THREADS;
            host::Block blk;
            blk.run(COOP_THREADS,
                    [&] {
                        if (rows <= 64)
                            base_block_coop_kernel<N, 2>(A.data(), n, n, 0, b, rows, ipiv.data(), &info, sc);
                        else
                            base_block_coop_kernel<N, 8>(A.data(), n, n, 0, b, rows, ipiv.data(), &info, sc);
                    },
                    make_order(order, seed + (uint64_t)k, COOP_THREADS / 32));
        });
    for (auto& t : blocks) t.join();
    printf("error %d info %d\npivots", sc->error, info);
    for (int v : ipiv) printf(" %d", v);
    printf("\nwords");
    for (double v : A) printf(" %a", v);
    printf("\n");
    delete sc;
}

int main(int argc, char** argv) {
    if (argc != 7) return 2;
    const int N = atoi(argv[1]), n = atoi(argv[2]), b = atoi(argv[3]), rows = atoi(argv[4]);
    const std::string order = argv[5];
    const uint64_t seed = strtoull(argv[6], nullptr, 10);
    if (b < 1 || b > PBASE || n < b || rows < 1 || rows > 256) return 2;
    if (N == 2) go<2>(n, b, rows, order, seed);
    else if (N == 3) go<3>(n, b, rows, order, seed);
    else if (N == 4) go<4>(n, b, rows, order, seed);
    else return 2;
    return 0;
}
