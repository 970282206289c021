// C ABI entry points, handle and device workspace.
#include <string.h>

#include <math.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>

#include "ozlu_internal.h"
#include "ozlu_handle.h"

namespace ozlu {

int cuda_rc(cudaError_t e) { return e == cudaSuccess ? OZLU_OK : OZLU_ERR_CUDA; }

namespace {
std::atomic<int> g_fail_allocs{0};  // allocations still to fail (test injection)
std::atomic<long long> g_alloc_limit{0};  // size from which allocations fail; 0: none (test injection)
std::mutex g_attr_mutex;
std::map<std::pair<const void*, int>, int> g_smem_set;  // (kernel, device) -> bytes set
constexpr int MAX_DEVICES = 64;
std::atomic<int> g_sms[MAX_DEVICES];
}  // namespace

bool dev_alloc(void** p, size_t bytes) {
    *p = nullptr;
    for (int v = g_fail_allocs.load(); v > 0; v = g_fail_allocs.load())
        if (g_fail_allocs.compare_exchange_weak(v, v - 1)) return false;
    const long long limit = g_alloc_limit.load();
    if (limit > 0 && bytes >= (size_t)limit) return false;
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    return true;
}

void raise_smem_limit(const void* kernel, int bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    std::lock_guard<std::mutex> lock(g_attr_mutex);
    auto key = std::make_pair(kernel, dev);
    auto it = g_smem_set.find(key);
    if (it != g_smem_set.end() && it->second >= bytes) return;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess)
        g_smem_set[key] = bytes;
    else
        cudaGetLastError();
}

int device_sms() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 1;
    if (dev < MAX_DEVICES) {
        const int v = g_sms[dev].load();
        if (v > 0) return v;
    }
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
    if (dev < MAX_DEVICES) g_sms[dev].store(sms);
    return sms;
}

bool is_device_ptr(const void* p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// the handle's device error word (OZLU_ERR_TIMEOUT from a bounded wait in a
// tensor-core GEMM); allocated once, zeroed in stream order by each call
int* err_word(ozlu_handle* h) {
    if (!h->dev_err) {
        if (!dev_alloc((void**)&h->dev_err, 256)) {
            h->dev_err = nullptr;
            return nullptr;
        }
        if (cudaMemsetAsync(h->dev_err, 0, 256, h->stream) != cudaSuccess) return nullptr;
    }
    return h->dev_err;
}

int clear_err_word(ozlu_handle* h) {
    int* e = err_word(h);
    if (!e) return OZLU_ERR_NOMEM;
    h->err_subs = 0;
    return cudaMemsetAsync(e, 0, sizeof(int), h->stream) == cudaSuccess ? OZLU_OK : OZLU_ERR_CUDA;
}

int finish_call(ozlu_handle* h) {
    int err = 0;
    if (h->dev_err && cudaMemcpyAsync(&err, h->dev_err, sizeof err, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
        return OZLU_ERR_CUDA;
    return cudaStreamSynchronize(h->stream) == cudaSuccess ? err : OZLU_ERR_CUDA;
}

int Workspace::ensure(size_t bytes) {
    if (bytes <= cap) return OZLU_OK;
    if (base) cudaFree(base);
    base = nullptr;
    cap = 0;
    ++moves;
    size_t want = bytes + bytes / 8;
    if (!dev_alloc(&base, want)) {
        if (!dev_alloc(&base, bytes)) {
            base = nullptr;
            return OZLU_ERR_NOMEM;
        }
        want = bytes;
    }
    cap = want;
    return OZLU_OK;
}

int ensure_unmoved(const ozlu_handle* h, Workspace& ws, size_t bytes) {
    return h->capturing && bytes > ws.cap ? RC_WOULD_MOVE : ws.ensure(bytes);
}

void Workspace::release() {
    if (base) cudaFree(base);
    base = nullptr;
    cap = 0;
}

int plan_for(ozlu_handle* h, int p, int K, const ozlu_opts* o, const PlanEntry** out) {
    ozlu_opts d;
    memset(&d, 0, sizeof d);
    if (!o) o = &d;
    auto key = std::make_tuple(p, K, o->backend, o->nslice, o->extra_groups, o->g_ex);
    auto it = h->plans.find(key);
    if (it == h->plans.end()) {
        PlanEntry e;
        int rc = make_plan(p, K, o, e.plan);
        if (rc) return rc;
        fill_table(e.plan, e.table);
        if (e.plan.backend != OZLU_BE_FP64) {
            fill_conv(e.table, e.conv);
            fill_crt(e.table, e.plan.pint_bits, e.crt);
            fill_gemm(e.table, e.plan.backend == OZLU_BE_FP8, e.gemm);
        }
        it = h->plans.emplace(key, e).first;
    }
    *out = &it->second;
    return OZLU_OK;
}

static size_t align_up(size_t v) { return (v + 255) / 256 * 256; }

// Measured choice of the residue back-end and the slice count (Sec. 3.5
// guideline: the format maximising bits per modulus times engine throughput,
// which the paper concludes can only be decided by measuring at the actual
// size; Sec. 3.2: S balances conversion against GEMM cost).  For each
// feasible back-end the slice counts tried are the smallest feasible S_min,
// S_min + 1 and the cost model's S* of Eq. (Lhint) when it is larger (only
// the caller's S when opts->nslice is set).  Every
// candidate whose model time (residue ops / engine rate) is within 4x of the
// best model is run on the caller's operands into a scratch C (once untimed,
// then twice timed with events, the faster counting); the fastest (back-end,
// S) is cached per (nc, p, k, options, log2 m, log2 n).  The first call of a
// new shape therefore waits for the stream.
int autotune(ozlu_handle* h, int nc, int p, int m, int n, int k, const double* A, long long lda,
             const double* B, long long ldb, const ozlu_opts& o, int* be_out, int* s_out) {
    auto lg = [](int v) { int r = 0; while ((1 << r) < v) ++r; return r; };
    const auto key = std::make_tuple(nc, p, k, o.nslice * 1000000 + o.extra_groups * 1000 + o.g_ex,
                                     lg(m), lg(n));
    auto it = h->tuned.find(key);
    if (it != h->tuned.end()) {
        *be_out = it->second.first;
        *s_out = it->second.second;
        return OZLU_OK;
    }
    // engine rates in residue-product tera-ops per second (GB300 measurements)
    // and the Eq. (Lhint) cost ratios r (the paper's 30 for INT8-class
    // engines, 17.9 for binary64)
    const int cand_be[4] = {OZLU_BE_FP16, OZLU_BE_FP8, OZLU_BE_INT8, OZLU_BE_FP64};
    const double rate[4] = {600.0, 1700.0 / 3.0, 600.0, 1.0};
    const double rcost[4] = {30.0, 30.0, 30.0, 17.9};
    struct Cand { int be, S; double model; };
    std::vector<Cand> cands;
    double best_model = 1e300;
    for (int c = 0; c < 4; ++c) {
        ozlu_opts t = o;
        t.backend = cand_be[c];
        Plan pl;
        if (make_plan(p, k, &t, pl) != OZLU_OK) continue;
        std::vector<int> slist{pl.S};
        if (o.nslice == 0) {
            const int slack = (int)ceil(log2(2.0 * k) - 1e-12) + 16 + o.g_ex;
            const int seed = std::max(pl.S, lhint_S(rcost[c], p + slack, m, n));
            slist = {pl.S, pl.S + 1};
            if (seed > pl.S + 1) slist.push_back(seed);
        }
        for (int S : slist) {
            ozlu_opts ts = t;
            ts.nslice = S;
            Plan ps;
            if (make_plan(p, k, &ts, ps) != OZLU_OK) continue;
            if (t.backend == OZLU_BE_INT8) {  // the FP16 candidate of this S, if any, runs the same kernels
                ozlu_opts tf = ts;
                tf.backend = OZLU_BE_FP16;
                Plan pf;
                if (make_plan(p, k, &tf, pf) == OZLU_OK) continue;
            }
            const double model = 2.0 * m * n * (double)k * ps.N * ps.pair_terms / (rate[c] * 1e12);
            cands.push_back({cand_be[c], S, model});
            best_model = std::min(best_model, model);
        }
    }
    // scratch C
    const size_t cbytes = sizeof(double) * nc * (size_t)m * n;
    int rc = h->tune_ws.ensure(cbytes);
    if (rc) return rc;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int choice = OZLU_BE_INT8, choice_s = 0;
    const bool timing = h->timing;
    h->timing = false;
    for (const Cand& cd : cands) {
        if (cd.model > 4.0 * best_model) continue;
        ozlu_opts t = o;
        t.backend = cd.be;
        t.nslice = cd.S;
        // an untimed first run (workspace growth, first launch of a kernel),
        // then the faster of two timed runs
        float cms = 1e30f;
        for (int rep = 0; rep < 3 && !rc; ++rep) {
            cudaEventRecord(e0, h->stream);
            rc = gemm_device(h, nc, p, m, n, k, 1, A, lda, B, ldb, 0, (double*)h->tune_ws.base, m, &t);
            cudaEventRecord(e1, h->stream);
            if (rc) break;
            cudaEventSynchronize(e1);
            float ms = 0;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0 && ms < cms) cms = ms;
        }
        if (rc == OZLU_ERR_UNSUPPORTED) {
            rc = OZLU_OK;
            continue;
        }
        if (rc) break;
        if (cms < best) { best = cms; choice = cd.be; choice_s = cd.S; }
    }
    h->timing = timing;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc && rc != OZLU_ERR_UNSUPPORTED) return rc;
    h->tuned[key] = std::make_pair(choice, choice_s);
    h->stats.last_backend = choice;
    *be_out = choice;
    *s_out = choice_s;
    return OZLU_OK;
}

// What gemm_device answers for these options at this K without running it: a
// plan exists (for the autotuner, on any back-end), or why not
int check_plan(ozlu_handle* h, int p, int K, const ozlu_opts* opts) {
    const PlanEntry* pe;
    if (opts && opts->backend != OZLU_BE_AUTO) return plan_for(h, p, K, opts, &pe);
    const int cand[4] = {OZLU_BE_FP16, OZLU_BE_FP8, OZLU_BE_FP64, OZLU_BE_INT8};
    int rc = OZLU_OK;
    for (int be : cand) {
        ozlu_opts o;
        memset(&o, 0, sizeof o);
        if (opts) o = *opts;
        o.backend = be;
        if (!(rc = plan_for(h, p, K, &o, &pe))) break;
    }
    return rc;
}

// The device part of one GEMM, all pointers on the device.

int gemm_device(ozlu_handle* h, int nc, int p, int m, int n, int k, int alpha, const double* A,
                long long lda, const double* B, long long ldb, int beta, double* C,
                long long ldc, const ozlu_opts* opts) {
    cudaStream_t s = h->stream;
    if (m == 0 || n == 0) return OZLU_OK;
    if (k == 0) {
        if (beta == 0) {
            for (int j = 0; j < n; ++j)
                if (cudaMemsetAsync(C + (long long)j * ldc * nc, 0, sizeof(double) * nc * m, s))
                    return OZLU_ERR_CUDA;
        }
        return OZLU_OK;
    }
    ozlu_opts o;
    memset(&o, 0, sizeof o);
    if (opts) o = *opts;
    if (o.backend == OZLU_BE_AUTO) {
        int S = 0;
        const int rc0 = autotune(h, nc, p, m, n, k, A, lda, B, ldb, o, &o.backend, &S);
        if (rc0) return rc0;
        if (o.nslice == 0) o.nslice = S;
    }
    const PlanEntry* pe;
    int rc = plan_for(h, p, k, &o, &pe);
    if (rc) return rc;
    const Plan* pl = &pe->plan;
    const DevTable* tab = &pe->table;
    const int be = pl->backend;
    const int Mpad = (m + 127) / 128 * 128, Npad = (n + 127) / 128 * 128;
    GemmLayout& L = h->last;
    L.m = m; L.n = n; L.k = k; L.Mpad = Mpad; L.Npad = Npad;
    L.N = pl->N; L.S = pl->S; L.G = pl->G; L.backend = be;
    // An INT8 plan's residue products run as binary16 ones on tcgen05 (mode 2),
    // exactly and to the same t values: residues up to 127 are binary16 numbers,
    // and sums longer than binary32 holds exactly are folded in parts.  The int8
    // tensor rate of this GPU is far below the binary16 one: TD, 1777 x 611 x
    // 389, 672 us for the products by mma.sync on int8 and 100 by this, 809 and
    // 225 in all; QD, 1024^3, 620 us in all by the FP8 plan, 480 by this.
    // mma.sync (mode 0) is left for where the larger residues do not fit in
    // memory, and for the allocation-free product's fixed scratch.
    int mode = be == OZLU_BE_FP8 ? 1 : be == OZLU_BE_FP64 ? 3 : 2;
    int Kpad = 0;
    bool pack = false;
    double residue_bytes = 0.0, t_bytes = 0.0;  // of the layout, for the counters
    auto layout = [&](bool narrow) -> size_t {
        if (narrow) mode = 0;
        const int P = mode == 1 ? 3 : 1, esz = mode == 2 ? 2 : (mode == 3 ? 8 : 1);
        // K padded to the GEMM's step: 64 elements (INT8, FP16; the binary64 kernel
        // takes any), 128 for FP8 (the accumulator conditions hold for the plan's 128)
        Kpad = mode == 1 ? pl->Kpad : (k + 63) / 64 * 64;
        L.Kpad = Kpad;
        L.mode = mode;
        size_t off = 0;
        L.mu = off; off = align_up(off + sizeof(int) * m);
        L.nu = off; off = align_up(off + sizeof(int) * n);
        L.ra = off; off = align_up(off + (size_t)pl->N * pl->S * P * Mpad * Kpad * esz);
        L.rb = off; off = align_up(off + (size_t)pl->N * pl->S * P * Npad * Kpad * esz);
        // t values: bytes, 32-bit words (binary64), or a word per triple of moduli
        pack = (mode == 1 || mode == 2) && tc05_packs(pe->gemm, Mpad, Npad);
        const size_t tval = pack ? 4 * (size_t)pe->gemm.NT : (size_t)pl->N * (mode == 3 ? 4 : 1);
        L.t = off;  off = align_up(off + (size_t)pl->G * tval * m * n);
        L.pack = pack;
        residue_bytes = (double)pl->N * pl->S * P * ((double)Mpad + Npad) * Kpad * esz;
        t_bytes = (double)pl->G * tval * m * n;
        return off;
    };
    memcpy(L.mod, pl->mod, sizeof L.mod);
    int* derr = err_word(h);
    if (!derr) return OZLU_ERR_NOMEM;
    if ((rc = fit_workspace(h, be == OZLU_BE_INT8, layout))) return rc;
    const int P = mode == 1 ? 3 : 1;
    char* base = (char*)h->ws.base;
    int* mu = (int*)(base + L.mu);
    int* nu = (int*)(base + L.nu);
    void* RA = base + L.ra;
    void* RB = base + L.rb;
    uint8_t* T = (uint8_t*)(base + L.t);
    const int prev = h->open_phase;
    h->phase(PH_CONVERT);
    launch_shifts(A, lda, m, B, ldb, n, nc, k, pl->Q, mu, nu, h->clear_err ? derr : nullptr, s);
    h->clear_err = false;
    if (mode == 3) {
        launch_convert64(A, lda, nc, m, k, false, mu, *tab, Kpad, Mpad, (double*)RA, s);
        launch_convert64(B, ldb, nc, k, n, true, nu, *tab, Kpad, Npad, (double*)RB, s);
    } else {
        launch_convert(A, lda, m, B, ldb, n, nc, k, mu, nu, pe->conv, Kpad, Mpad, Npad, RA, RB, mode, s);
    }
    h->phase(PH_GEMM);
    if (mode == 0) {
        launch_gemm_imma((const int8_t*)RA, (const int8_t*)RB, m, n, Mpad, Npad, Kpad, *tab, T, s);
    } else if (mode == 3) {
        launch_gemm_f64((const double*)RA, (const double*)RB, m, n, Mpad, Npad, Kpad, *tab, (uint32_t*)T, s);
    } else {
        rc = launch_gemm_tc05(mode == 1, pack, RA, RB, m, n, Mpad, Npad, Kpad, pe->gemm, T, derr, s);
        if (rc) return rc;
    }
    h->phase(PH_CRT);
    if (mode == 3) launch_crt64((const uint32_t*)T, m, n, mu, nu, *tab, nc, alpha, beta, C, ldc, s);
    else launch_crt(T, pack, m, n, mu, nu, pe->crt, nc, alpha, beta, C, ldc, s);
    h->phase(prev);
    h->stats.gemm_launches += 1;
    h->stats.crt_launches += 1;
    h->stats.last_backend = be;
    h->stats.last_nslice = pl->S;
    h->stats.gemm_ops += 2.0 * m * n * (double)k * pl->N * pl->pair_terms * P;
    h->stats.crt_bytes += t_bytes + 8.0 * nc * m * n * (beta ? 2 : 1);
    h->stats.convert_bytes += 8.0 * nc * ((double)m * k + (double)k * n) + residue_bytes;
    h->count(mode == 3 ? 5 : 4);
    if (cudaGetLastError() != cudaSuccess) return OZLU_ERR_CUDA;
    return OZLU_OK;
}

}  // namespace ozlu

void ozlu_handle::phase(int ph) {
    if (!timing) return;
    if (open_phase >= 0) {
        if (pool_used == pool.size()) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            pool.push_back(e);
        }
        cudaEvent_t end = pool[pool_used++];
        cudaEventRecord(end, stream);
        marks.push_back({open_phase, {open_ev, end}});
    }
    open_phase = ph;
    if (ph >= 0) {
        if (pool_used == pool.size()) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            pool.push_back(e);
        }
        open_ev = pool[pool_used++];
        cudaEventRecord(open_ev, stream);
    }
}

void ozlu_handle::resolve_times() {
    if (marks.empty()) return;
    cudaEventSynchronize(marks.back().second.second);
    for (auto& mk : marks) {
        float ms = 0;
        cudaEventElapsedTime(&ms, mk.second.first, mk.second.second);
        double* dst[] = {&stats.convert_ms, &stats.gemm_ms, &stats.crt_ms, &stats.panel_ms,
                         &stats.other_ms, &stats.trsm_ms};
        *dst[mk.first] += ms;
    }
    marks.clear();
    pool_used = open_phase >= 0 ? pool_used : 0;
}

using namespace ozlu;

extern "C" {

const char* ozlu_version(void) { return "ozlu 0.2 (sm_103a)"; }

int ozlu_debug_fail_alloc(int count) {
    if (count < 0) return -1;
    g_fail_allocs.store(count);
    return OZLU_OK;
}

int ozlu_debug_limit_alloc(long long bytes) {
    if (bytes < 0) return -1;
    g_alloc_limit.store(bytes);
    return OZLU_OK;
}

int ozlu_create(ozlu_handle** handle, void* stream) {
    if (!handle) return -1;
    *handle = nullptr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return OZLU_ERR_CUDA;
    }
    ozlu_handle* h = new ozlu_handle();
    h->device = dev;
    h->stream = (cudaStream_t)stream;
    *handle = h;
    return OZLU_OK;
}

int ozlu_destroy(ozlu_handle* h) {
    if (!h) return OZLU_OK;
    cudaStreamSynchronize(h->stream);
    for (auto& g : h->graphs)
        if (g.second.exec) cudaGraphExecDestroy(g.second.exec);
    h->graphs.clear();
    for (int k = 0; k < MAX_SUB; ++k) {
        if (h->sub[k]) {
            cudaStream_t s = h->sub[k]->stream;
            ozlu_destroy(h->sub[k]);
            cudaStreamDestroy(s);
        }
        if (h->join[k]) cudaEventDestroy(h->join[k]);
    }
    if (h->fork) cudaEventDestroy(h->fork);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    if (h->dev_err) cudaFree(h->dev_err);
    for (auto& e : h->ext_plans)
        if (e.second.dev) cudaFree(e.second.dev);
    h->ext_plans.clear();
    h->ws.release();
    h->stage.release();
    h->tune_ws.release();
    h->solve_ws.release();
    h->nb_ws.release();
    if (h->lu_scratch) cudaFree(h->lu_scratch);
    if (h->coop_scratch) cudaFree(h->coop_scratch);
    for (auto& e : h->pool) cudaEventDestroy(e);
    delete h;
    return OZLU_OK;
}

int ozlu_debug_wait_limit(ozlu_handle* h, long long limit) {
    if (!h) return -1;
    if (limit < 0) return -2;
    h->wait_limit = limit;
    return OZLU_OK;
}

int ozlu_set_stream(ozlu_handle* h, void* stream) {
    if (!h) return -1;
    h->stream = (cudaStream_t)stream;
    return OZLU_OK;
}

int ozlu_set_timing(ozlu_handle* h, int enable) {
    if (!h) return -1;
    for (int k = 0; k < MAX_SUB; ++k)
        if (h->sub[k]) ozlu_set_timing(h->sub[k], enable);
    h->phase(-1);
    h->resolve_times();
    h->timing = enable != 0;
    memset(&h->stats, 0, sizeof h->stats);
    return OZLU_OK;
}

// the handle's counters plus those of its batched-driver sub-handles (phase
// times of concurrent sub-streams add up, so they may exceed the wall time)
int ozlu_get_stats(ozlu_handle* h, ozlu_stats* out) {
    if (!h) return -1;
    if (!out) return -2;
    h->phase(-1);
    h->resolve_times();
    *out = h->stats;
    for (int k = 0; k < MAX_SUB; ++k) {
        ozlu_handle* s = h->sub[k];
        if (!s) continue;
        s->phase(-1);
        s->resolve_times();
        const ozlu_stats& d = s->stats;
        out->convert_ms += d.convert_ms;
        out->gemm_ms += d.gemm_ms;
        out->crt_ms += d.crt_ms;
        out->panel_ms += d.panel_ms;
        out->other_ms += d.other_ms;
        out->trsm_ms += d.trsm_ms;
        out->gemm_launches += d.gemm_launches;
        out->crt_launches += d.crt_launches;
        out->panel_launches += d.panel_launches;
        out->launches += d.launches;
        out->gemm_ops += d.gemm_ops;
        out->crt_bytes += d.crt_bytes;
        out->convert_bytes += d.convert_bytes;
        if (d.last_backend) out->last_backend = d.last_backend;
    }
    return OZLU_OK;
}

int ozlu_gemm(ozlu_handle* h, int nc, int p, int m, int n, int k, int alpha, const double* A,
              long long lda, const double* B, long long ldb, int beta, double* C, long long ldc,
              const ozlu_opts* opts) {
    if (!h) return -1;
    if (nc < 2 || nc > 4) return -2;
    if (p == 0) p = 53 * nc;
    if (p < 1 || p > 53 * nc) return -3;
    if (m < 0) return -4;
    if (n < 0) return -5;
    if (k < 0) return -6;
    if (alpha != 1 && alpha != -1) return -7;
    if (!A && m && k) return -8;
    if (lda < (m > 1 ? m : 1)) return -9;
    if (!B && k && n) return -10;
    if (ldb < (k > 1 ? k : 1)) return -11;
    if (beta != 0 && beta != 1) return -12;
    if (!C && m && n) return -13;
    if (ldc < (m > 1 ? m : 1)) return -14;
    if (cudaSetDevice(h->device) != cudaSuccess) return OZLU_ERR_CUDA;
    // the product's first kernel clears the error word, or this where none runs
    if (!err_word(h)) return OZLU_ERR_NOMEM;
    auto product = [&](const double* a, const double* b, double* c) -> int {
        h->clear_err = true;
        h->err_subs = 0;
        const int rc = gemm_device(h, nc, p, m, n, k, alpha, a, lda, b, ldb, beta, c, ldc, opts);
        const int rc1 = h->clear_err ? clear_err_word(h) : OZLU_OK;
        h->clear_err = false;
        return rc ? rc : rc1;
    };
    const bool dA = !A || is_device_ptr(A), dB = !B || is_device_ptr(B), dC = !C || is_device_ptr(C);
    if (dA && dB && dC) return product(A, B, C);
    // stage host operands through a second device buffer
    const size_t ea = (size_t)lda * (k ? k : 1) * nc, eb = (size_t)ldb * (n ? n : 1) * nc,
                 ec = (size_t)ldc * (n ? n : 1) * nc;
    const size_t bytes = sizeof(double) * (ea + eb + ec) + 3 * 256;
    int rc = h->stage.ensure(bytes);
    if (rc) return rc;
    double* sA = (double*)h->stage.base;
    double* sB = (double*)((char*)sA + align_up(sizeof(double) * ea));
    double* sC = (double*)((char*)sB + align_up(sizeof(double) * eb));
    cudaStream_t s = h->stream;
    const double* gA = A;
    const double* gB = B;
    double* gC = C;
    if (!dA) { if (cudaMemcpyAsync(sA, A, sizeof(double) * ea, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA; gA = sA; }
    if (!dB) { if (cudaMemcpyAsync(sB, B, sizeof(double) * eb, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA; gB = sB; }
    if (!dC) {
        if (beta && cudaMemcpyAsync(sC, C, sizeof(double) * ec, cudaMemcpyHostToDevice, s)) return OZLU_ERR_CUDA;
        gC = sC;
    }
    rc = product(gA, gB, gC);
    if (rc) return rc;
    if (!dC && cudaMemcpyAsync(C, sC, sizeof(double) * ec, cudaMemcpyDeviceToHost, s)) return OZLU_ERR_CUDA;
    return finish_call(h);
}

int ozlu_debug_fetch(ozlu_handle* h, int what, void* dst, size_t bytes) {
    if (!h) return -1;
    if (!dst) return -3;
    const GemmLayout& L = h->last;
    char* base = (char*)h->ws.base;
    if (what == 6) {
        if (bytes < sizeof(int)) return -4;
        if (cudaStreamSynchronize(h->stream)) return OZLU_ERR_CUDA;
        // the handle's own word, or those of the sub-handles that ran its last call
        int err = 0;
        for (int k = -1; k < MAX_SUB && !err; ++k) {
            ozlu_handle* s = k < 0 ? (h->err_subs ? nullptr : h) : (h->err_subs >> k & 1 ? h->sub[k] : nullptr);
            if (s && s->dev_err && cudaMemcpy(&err, s->dev_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
                return OZLU_ERR_CUDA;
        }
        *(int*)dst = err;
        return OZLU_OK;
    }
    if (!base) return OZLU_ERR_CAPACITY;
    if (cudaStreamSynchronize(h->stream)) return OZLU_ERR_CUDA;
    if (what == 1 || what == 2) {
        const size_t need = sizeof(int) * (what == 1 ? L.m : L.n);
        if (bytes < need) return -4;
        return cuda_rc(cudaMemcpy(dst, base + (what == 1 ? L.mu : L.nu), need, cudaMemcpyDeviceToHost));
    }
    if ((what == 3 || what == 4) && L.backend != OZLU_BE_INT8) return OZLU_ERR_UNSUPPORTED;
    if (what == 3 || what == 4) {
        const int R = what == 3 ? L.m : L.n, Rpad = what == 3 ? L.Mpad : L.Npad;
        const size_t need = (size_t)L.N * L.S * R * L.k;
        if (bytes < need) return -4;
        const char* src = base + (what == 3 ? L.ra : L.rb);
        if (L.mode == 2) {  // binary16 encodings of the same residues
            std::vector<uint16_t> row((size_t)R * L.k);
            for (int pl = 0; pl < L.N * L.S; ++pl) {
                if (cudaMemcpy2D(row.data(), 2 * (size_t)L.k, src + 2 * (size_t)pl * Rpad * L.Kpad,
                                 2 * (size_t)L.Kpad, 2 * (size_t)L.k, R, cudaMemcpyDeviceToHost) != cudaSuccess)
                    return OZLU_ERR_CUDA;
                int8_t* out = (int8_t*)dst + (size_t)pl * R * L.k;
                for (size_t e = 0; e < row.size(); ++e) {
                    const int ex = (row[e] >> 10) & 31, fr = (row[e] & 0x3ff) | 0x400;
                    const int v = ex ? fr >> (25 - ex) : 0;  // an integer below 128
                    out[e] = (int8_t)(row[e] >> 15 ? -v : v);
                }
            }
            return OZLU_OK;
        }
        for (int pl = 0; pl < L.N * L.S; ++pl)
            if (cudaMemcpy2D((char*)dst + (size_t)pl * R * L.k, L.k, src + (size_t)pl * Rpad * L.Kpad,
                             L.Kpad, L.k, R, cudaMemcpyDeviceToHost) != cudaSuccess)
                return OZLU_ERR_CUDA;
        return OZLU_OK;
    }
    if (what == 5) {
        const size_t need = (size_t)L.G * L.N * L.m * L.n * (L.backend == OZLU_BE_FP64 ? 4 : 1);
        if (bytes < need) return -4;
        if (!L.pack) return cuda_rc(cudaMemcpy(dst, base + L.t, need, cudaMemcpyDeviceToHost));
        // a packed word u = t_a m_b m_c + t_b m_a m_c + t_c m_a m_b gives
        // t_a = u (m_b m_c)^-1 mod m_a
        const size_t mn = (size_t)L.m * L.n;
        const int NT = (L.N + 2) / 3;
        std::vector<uint32_t> u(mn);
        for (int gi = 0; gi < L.G; ++gi)
            for (int q = 0; q < NT; ++q) {
                if (cudaMemcpy(u.data(), base + L.t + 4 * mn * ((size_t)gi * NT + q), 4 * mn,
                               cudaMemcpyDeviceToHost) != cudaSuccess)
                    return OZLU_ERR_CUDA;
                for (int l = 3 * q; l < 3 * q + 3 && l < L.N; ++l) {
                    const uint32_t ml = (uint32_t)L.mod[l];
                    uint32_t others = 1, inv = 1;
                    for (int j = 3 * q; j < 3 * q + 3 && j < L.N; ++j)
                        if (j != l) others = others * (uint32_t)L.mod[j] % ml;
                    while (others * inv % ml != 1 % ml) ++inv;
                    uint8_t* out = (uint8_t*)dst + mn * ((size_t)gi * L.N + l);
                    for (size_t e = 0; e < mn; ++e) out[e] = (uint8_t)(u[e] % ml * inv % ml);
                }
            }
        return OZLU_OK;
    }
    return -2;
}

}  // extern "C"
