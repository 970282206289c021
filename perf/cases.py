"""What the framework's users have it do, as cases that can be timed.

Every case goes through a public entry point of paper_2609_29554_gb300.ozlu with
matrices in device memory, as a program calls it: the Ozaki-II GEMM in
double-, triple- and quad-double (DD, TD, QD), its allocation-free form, the LU
factorisation (one matrix, a batch of uneven ones), the solve, and the p-bit
GEMM and LU.  A program keeps one handle for its life, so the cases share one;
matrices that a call overwrites are restored by a device copy inside the pass,
which is what a program that factors again and again pays too.
"""
import math

import torch

from paper_2609_29554_gb300 import ozlu

_HANDLE = None


def _handle():
    global _HANDLE
    if _HANDLE is None:
        torch.cuda.init()
        _HANDLE = ozlu.ozlu_create(None)
    return _HANDLE


# ------------------------------------------------------------------- the cases
def _gemm(m, n, k, nc, alpha=1, beta=0, backend="auto", pad=0):
    return {"kind": "gemm", "m": m, "n": n, "k": k, "nc": nc, "alpha": alpha, "beta": beta,
            "backend": backend, "pad": pad}


def _lu(n, nc, nb, cond, backend="auto", graph=0):
    return {"kind": "lu", "n": n, "nc": nc, "nb": nb, "cond": cond, "backend": backend, "graph": graph}


def listed():
    def named(name, c):
        return dict(c, name=name)

    return [
        # a small product inside a larger program: latency and launches
        named("gemm_dd_32", _gemm(32, 32, 32, 2)),
        # the same for a caller that must not allocate, as an update C <- C - A B
        named("noalloc_qd_96", {"kind": "noalloc", "m": 96, "n": 96, "k": 96, "nc": 4}),
        # the standalone QD product at the smallest size of its benchmark
        named("gemm_qd_1024", _gemm(1024, 1024, 1024, 4)),
        # a ragged TD product with leading dimensions of its own, INT8 residues
        # (the default of make_opts)
        named("gemm_td_ragged_int8", _gemm(1777, 611, 389, 3, backend="int8", pad=7)),
        # the trailing update of the first step of the n = 4096 LU with nb = 256
        named("gemm_qd_update_3840", _gemm(3840, 3840, 256, 4, alpha=-1, beta=1)),
        # the small LU: n = 128, panels of 32 columns, INT8 residues
        named("lu_dd_128_nb32", _lu(128, 2, 32, 0, "int8")),
        # a mid-size LU of a well-conditioned matrix, called directly
        named("lu_qd_1000", _lu(1000, 4, 256, 0)),
        # the headline LU: cond 1e40, replayed as a CUDA graph
        named("lu_qd_4096_graph", _lu(4096, 4, 256, 40, graph=1)),
        # many uneven systems at once: LU and solve of a batch, as CUDA graphs
        named("batched_td_48", {"kind": "batched", "count": 48, "nmin": 64, "nmax": 768, "nc": 3}),
        # a solve from factors that are kept
        named("solve_qd_1500", {"kind": "solve", "n": 1500, "nrhs": 3, "nc": 4}),
        # p-bit arithmetic: the product, and an LU with its solve
        named("mp_gemm_1024b_512", {"kind": "mp_gemm", "m": 512, "n": 512, "k": 512, "p": 1024}),
        named("mp_lu_1216b_192", {"kind": "mp_lu", "n": 192, "p": 1216, "nrhs": 1}),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "noalloc", "lu", "lu", "batched", "solve", "mp_gemm", "mp_lu"])
    nc = rng.choice([2, 3, 4])
    if kind == "gemm":
        # products from a few rows to the benchmark's sizes, wide and narrow ones
        m, n = _logint(rng, 16, 3000), _logint(rng, 16, 3000)
        k = _logint(rng, 16, 1500)
        beta = rng.choice([0, 1])
        return _gemm(m, n, k, nc, alpha=-1 if beta else 1, beta=beta,
                     backend=rng.choice(["auto", "auto", "int8"]), pad=rng.choice([0, 0, 5]))
    if kind == "noalloc":
        return {"kind": kind, "m": _logint(rng, 8, 128), "n": _logint(rng, 8, 128),
                "k": _logint(rng, 8, 128), "nc": nc}
    if kind == "lu":
        n = _logint(rng, 48, 2048)
        return _lu(n, nc, rng.choice([32, 64, 128, 256]), rng.choice([0, 0, 5 * nc]),
                   rng.choice(["auto", "auto", "int8"]), rng.choice([0, 1]))
    if kind == "batched":
        lo = _logint(rng, 16, 128)
        return {"kind": kind, "count": rng.randint(2, 40), "nmin": lo, "nmax": lo + rng.randint(8, 500), "nc": nc}
    if kind == "solve":
        return {"kind": kind, "n": _logint(rng, 40, 2048), "nrhs": _logint(rng, 1, 64), "nc": nc}
    if kind == "mp_gemm":
        return {"kind": kind, "m": _logint(rng, 8, 400), "n": _logint(rng, 8, 400),
                "k": _logint(rng, 8, 400), "p": _logint(rng, 128, 2048)}
    n = _logint(rng, 16, 160)
    return {"kind": kind, "n": n, "p": 64 * math.ceil(1.2 * 5.1 * n / 64), "nrhs": rng.choice([1, 1, 4])}


# ------------------------------------------------------------------ the inputs
def _pow2(e):
    """2^e exactly (float64), e an int64 tensor in the normal range."""
    return ((e + 1023) << 52).view(torch.float64)


def _lift(lead, nc, gen):
    """Expansions with the given leading components: each lower component is
    random below a quarter ulp of the one before it, so that the leading one is
    the rounded value."""
    out = torch.zeros(lead.shape + (nc,), dtype=torch.float64, device="cuda")
    out[..., 0] = lead
    for c in range(1, nc):
        e = torch.frexp(out[..., c - 1])[1].to(torch.int64)
        u = 2.0 * torch.rand(lead.shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0
        out[..., c] = torch.where(out[..., c - 1] != 0, u * _pow2((e - 55).clamp(min=-1000)), torch.zeros_like(u))
    return out


def _uniform(shape, gen):
    return 2.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0


def _random_matrix(rows, cols, ld, nc, spread, gen):
    """(cols, ld, nc): uniform [-1, 1) leading components times 2^e, e uniform in
    [-spread, spread] (the standalone product's entries have spread 30)."""
    lead = _uniform((cols, ld), gen)
    if spread:
        e = torch.randint(-spread, spread + 1, (cols, ld), device="cuda", generator=gen)
        lead = lead * _pow2(e)
    lead[:, rows:] = 0.0
    return _lift(lead, nc, gen)


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _ill_conditioned(n, nc, log10_cond, gen):
    """(n, n, nc): G diag(sigma) H, G and H seeded normal matrices on the grid
    2^-21, sigma geometric from 1 to 10^-log10_cond (powers of two).  The
    product is summed exactly per exponent (integers below 2^53) and the
    exponents are accumulated in nc + 1 components, so the small singular
    values survive."""
    def grid():
        z = torch.randn((n, n), dtype=torch.float64, device="cuda", generator=gen)
        return torch.round((z / math.sqrt(n)).clamp(-0.99, 0.99) * 2.0 ** 21)

    G, H = grid(), grid()
    k = torch.arange(n, dtype=torch.float64)
    e = torch.round(-math.log2(10.0) * log10_cond * k / max(n - 1, 1)).to(torch.int64).tolist()
    acc = [torch.zeros((n, n), dtype=torch.float64, device="cuda") for _ in range(nc + 1)]
    k0 = 0
    while k0 < n:
        k1 = k0
        while k1 < n and e[k1] == e[k0] and k1 - k0 < 512:
            k1 += 1
        t = (H[:, k0:k1] @ G[k0:k1]) * 2.0 ** (e[k0] - 42)
        for c in range(nc + 1):
            acc[c], t = _two_sum(acc[c], t)
        k0 = k1
    for _ in range(nc + 1):
        for c in range(nc - 1, -1, -1):
            acc[c], acc[c + 1] = _two_sum(acc[c], acc[c + 1])
    return torch.stack(acc[:nc], dim=-1).contiguous()


def _lu_matrix(n, nc, cond, gen):
    return _ill_conditioned(n, nc, cond, gen) if cond else _random_matrix(n, n, n, nc, 0, gen)


def _mp_random(rows, cols, L, gen, spread=8):
    M = ozlu.MPMatrix(rows, cols, L)
    lim = torch.randint(0, 1 << 32, (L, rows * cols), device="cuda", generator=gen)
    lim[L - 1] |= 1 << 31
    M.limbs.copy_(torch.where(lim >= 1 << 31, lim - (1 << 32), lim).to(torch.int32))
    M.exps.copy_(torch.randint(-spread, spread + 1, (rows * cols,), device="cuda", generator=gen))
    M.signs.copy_(torch.randint(0, 2, (rows * cols,), device="cuda", generator=gen))
    return M


def _mp_copy(dst, src):
    dst.limbs.copy_(src.limbs)
    dst.exps.copy_(src.exps)
    dst.signs.copy_(src.signs)


def _batch_sizes(c):
    """The batch's sizes: fixed by the case, spread over [nmin, nmax]."""
    span, cnt = c["nmax"] - c["nmin"], c["count"]
    return [c["nmin"] + (span * ((i * 7919) % cnt) + (i * 31) % max(span, 1)) // cnt % (span + 1) for i in range(cnt)]


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    h = _handle()
    kind = c["kind"]
    s = {"case": c, "h": h}
    if kind in ("gemm", "noalloc"):
        m, n, k, nc, pad = c["m"], c["n"], c["k"], c["nc"], c.get("pad", 0)
        update = kind == "noalloc" or c["beta"]
        spread = 3 if update else 30  # an update's operands are factors of one matrix
        s["lda"], s["ldb"], s["ldc"] = m + pad, k + pad, m + pad
        s["A"] = _random_matrix(m, k, s["lda"], nc, spread, gen)
        s["B"] = _random_matrix(k, n, s["ldb"], nc, spread, gen)
        s["C0"] = _random_matrix(m, n, s["ldc"], nc, spread, gen) if update else None
        s["C"] = torch.zeros((n, s["ldc"], nc), dtype=torch.float64, device="cuda")
        if kind == "gemm":
            s["opts"] = ozlu.make_opts(c["backend"])
    elif kind == "lu":
        n, nc = c["n"], c["nc"]
        s["A"] = _lu_matrix(n, nc, c["cond"], gen)
        s["LU"] = torch.empty_like(s["A"])
        s["ipiv"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["info"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        s["opts"] = ozlu.make_opts(c["backend"], graph=c["graph"])
    elif kind == "batched":
        nc, ns = c["nc"], _batch_sizes(c)
        mats = [_lu_matrix(n, nc, 0, gen).reshape(-1) for n in ns]
        s["A"] = torch.cat(mats)
        s["LU"] = torch.empty_like(s["A"])
        s["B"] = _random_matrix(sum(ns), 1, sum(ns), nc, 0, gen)
        s["X"] = torch.empty_like(s["B"])
        s["ipiv"] = torch.zeros(sum(ns), dtype=torch.int32, device="cuda")
        s["info"] = torch.zeros(len(ns), dtype=torch.int32, device="cuda")
        s["ns"] = ns
        s["mats"] = list(s["LU"].split([n * n * nc for n in ns]))
        s["pivs"] = list(s["ipiv"].split(ns))
        s["xs"] = list(s["X"].reshape(-1).split([n * nc for n in ns]))
        s["opts"] = ozlu.make_opts("auto", graph=1)
    elif kind == "solve":
        n, nc, nrhs = c["n"], c["nc"], c["nrhs"]
        lu, piv = torch.linalg.lu_factor(_uniform((n, n), gen))
        s["LU"] = _lift(lu.T.contiguous(), nc, gen)
        s["ipiv"] = piv.to(torch.int32)
        s["B"] = _random_matrix(n, nrhs, n, nc, 0, gen)
        s["X"] = torch.empty_like(s["B"])
    elif kind == "mp_gemm":
        L = (c["p"] + 31) // 32
        s["A"] = _mp_random(c["m"], c["k"], L, gen)
        s["B"] = _mp_random(c["k"], c["n"], L, gen)
        s["C"] = ozlu.MPMatrix(c["m"], c["n"], L)
    else:
        n, L = c["n"], (c["p"] + 31) // 32
        s["A"] = _mp_random(n, n, L, gen, 1)
        s["LU"] = ozlu.MPMatrix(n, n, L)
        s["B"] = _mp_random(n, c["nrhs"], L, gen, 1)
        s["X"] = ozlu.MPMatrix(n, c["nrhs"], L)
        s["ipiv"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["info"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


# ---------------------------------------------------------------------- a pass
def run(s):
    c, h = s["case"], s["h"]
    kind = c["kind"]
    if kind in ("gemm", "noalloc"):
        if s["C0"] is not None:
            s["C"].copy_(s["C0"])
        if kind == "noalloc":
            ozlu.ozlu_gemm_noalloc(c["nc"], 0, c["m"], c["n"], c["k"], -1, s["A"], s["lda"], s["B"], s["ldb"],
                                   1, s["C"], s["ldc"])
        else:
            ozlu.ozlu_gemm(h, c["nc"], 0, c["m"], c["n"], c["k"], c["alpha"], s["A"], s["lda"], s["B"], s["ldb"],
                           c["beta"], s["C"], s["ldc"], s["opts"])
        return s["C"]
    if kind == "lu":
        s["LU"].copy_(s["A"])
        ozlu.ozlu_getrf(h, c["nc"], 0, c["n"], s["LU"], c["n"], s["ipiv"], c["nb"], s["info"], s["opts"])
        return {"LU": s["LU"], "ipiv": s["ipiv"], "info": s["info"]}
    if kind == "batched":
        s["LU"].copy_(s["A"])
        s["X"].copy_(s["B"])
        ozlu.ozlu_getrf_batched(h, c["nc"], 0, s["ns"], s["mats"], s["ns"], s["pivs"], s["info"], 128, s["opts"])
        ozlu.ozlu_getrs_batched(h, c["nc"], 0, s["ns"], 1, s["mats"], s["ns"], s["pivs"], s["xs"], s["ns"],
                                s["opts"])
        return {"LU": s["LU"], "X": s["X"], "ipiv": s["ipiv"], "info": s["info"]}
    if kind == "solve":
        s["X"].copy_(s["B"])
        ozlu.ozlu_getrs(h, c["nc"], 0, c["n"], c["nrhs"], s["LU"], c["n"], s["ipiv"], s["X"], c["n"])
        return s["X"]
    if kind == "mp_gemm":
        ozlu.ozlu_mp_gemm(h, c["p"], c["m"], c["n"], c["k"], 1, s["A"].desc(), s["B"].desc(), 0, s["C"].desc())
        return _mp_out(s["C"])
    _mp_copy(s["LU"], s["A"])
    _mp_copy(s["X"], s["B"])
    ozlu.ozlu_mp_getrf(h, c["p"], c["n"], s["LU"].desc(), s["ipiv"], 0, s["info"])
    ozlu.ozlu_mp_getrs(h, c["p"], c["n"], c["nrhs"], s["LU"].desc(), s["ipiv"], s["X"].desc())
    return {"LU": _mp_out(s["LU"]), "X": _mp_out(s["X"]), "ipiv": s["ipiv"], "info": s["info"]}


def _mp_out(M):
    return {"limbs": M.limbs, "exps": M.exps, "signs": M.signs}


# ------------------------------------------------------------------- its work
def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: the exact
    products of p-bit numbers as 8-bit residues, (2 p + log2 k) / 8 of them per
    multiply-add at the least."""
    c = case
    kind = c["kind"]

    def res(p, k):
        return math.ceil((2 * p + math.log2(max(k, 1))) / 8)

    def mb(p):
        return 4 * ((p + 31) // 32) + 8

    if kind in ("gemm", "noalloc"):
        m, n, k, nc = c["m"], c["n"], c["k"], c["nc"]
        upd = kind == "noalloc" or c["beta"]
        return {"bytes": 8 * nc * (m * k + k * n + m * n * (2 if upd else 1)), "flops": 2 * m * n * k * res(53 * nc, k)}
    if kind == "lu":
        n, nc = c["n"], c["nc"]
        return {"bytes": 16 * nc * n * n + 4 * n, "flops": 2 * n ** 3 / 3 * res(53 * nc, n)}
    if kind == "batched":
        ns, nc = _batch_sizes(c), c["nc"]
        return {"bytes": sum(16 * nc * (n * n + n) + 4 * n for n in ns),
                "flops": sum((2 * n ** 3 / 3 + 2 * n * n) * res(53 * nc, n) for n in ns)}
    if kind == "solve":
        n, nc, r = c["n"], c["nc"], c["nrhs"]
        return {"bytes": 8 * nc * (n * n + 2 * n * r) + 4 * n, "flops": 2 * n * n * r * res(53 * nc, n)}
    if kind == "mp_gemm":
        m, n, k, p = c["m"], c["n"], c["k"], c["p"]
        return {"bytes": mb(p) * (m * k + k * n + m * n), "flops": 2 * m * n * k * res(p, k)}
    n, p, r = c["n"], c["p"], c["nrhs"]
    return {"bytes": mb(p) * (2 * n * n + 2 * n * r) + 4 * n, "flops": (2 * n ** 3 / 3 + 2 * n * n * r) * res(p, n)}


# ---------------------------------------------------- the same in 64 bits
def _expand(lead, nc):
    """The 64-bit value laid out as an expansion: the lower components, below
    2^-53 of it, as zeros."""
    out = torch.zeros(lead.shape + (nc,), dtype=torch.float64, device=lead.device)
    out[..., 0] = lead
    return out


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind in ("mp_gemm", "mp_lu"):
        return None  # limbs: whole numbers
    if kind == "lu" and c["cond"]:
        return None  # 64 bits cannot factor a matrix of this condition
    s = prepare(case, seed)
    if kind in ("gemm", "noalloc"):
        nc = c["nc"]
        v = s["B"][:, :c["k"], 0] @ s["A"][:, :, 0]      # (n, k) (k, lda): column-major C
        if s["C0"] is not None:
            sign = -1.0 if kind == "noalloc" else float(c["alpha"])
            v = s["C0"][:, :, 0] + sign * v
        v[:, c["m"]:] = 0.0
        return _expand(v, nc)
    if kind == "lu":
        lu, piv = torch.linalg.lu_factor(s["A"][:, :, 0].T)
        return {"LU": _expand(lu.T, c["nc"]), "ipiv": None, "info": None}
    if kind == "solve":
        x = torch.linalg.lu_solve(s["LU"][:, :, 0].T.contiguous(), s["ipiv"], s["B"][:, :, 0].T.contiguous())
        return _expand(x.T, c["nc"])
    nc, lus, xs, at, row = c["nc"], [], [], 0, 0
    for n in s["ns"]:
        A = s["A"][at:at + n * n * nc].reshape(n, n, nc)[:, :, 0].T.contiguous()
        lu, piv = torch.linalg.lu_factor(A)
        lus.append(_expand(lu.T.contiguous(), nc).reshape(-1))
        xs.append(torch.linalg.lu_solve(lu, piv, s["B"][0, row:row + n, 0].reshape(n, 1))[:, 0])
        at += n * n * nc
        row += n
    return {"LU": torch.cat(lus), "X": _expand(torch.cat(xs), nc)[None], "ipiv": None, "info": None}
