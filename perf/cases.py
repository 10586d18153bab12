"""The work that users of this library have it do, as timed cases.

A case is a dict of plain values; ``listed`` gives the fixed ones, ``draw`` one
more of the same ranges, ``prepare`` what a program has in hand before the
call, ``run`` one pass through the public entry points, ``work`` the bytes and
operations the pass cannot do without, ``exact`` the same outputs by plain
torch and numpy in 64 bits, and ``tolerance`` how far another correct
implementation of the same precision may be from this one.

Handles are used as ``gbr_*_create`` returns them (no autotuning), since that is
what a program gets that only follows the header.
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_2203_04158_gb300 as G

LARGEST_HV = 11440 * 11440      # states of the largest H·v case (4x4 torus, 7 + 7 particles)


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # Ranking as a step of its own (a basis look-up service for another code's
        # states): the half-filled sector of 32 orbitals, where tables are largest.
        dict(name="comb_rank_m32", kind="comb_rank", M=32, N=16, n=1 << 27, bits=32, check=0),
        # The other direction: bit patterns of given indices, e.g. to enumerate or
        # sample a sector on the device.  Odd count.
        dict(name="comb_unrank_m32", kind="comb_unrank", M=32, N=16, n=(1 << 25) + 7, bits=32),
        # A set with no closed form of its index: two million 40-bit states, looked
        # up in random order, a ragged number of queries with strangers among them.
        dict(name="trie_rank_40bit", kind="trie_rank", width=40, members=1 << 21, n=(1 << 24) + 77, bits=32,
             check=1, msb=False),
        # The smallest H·v in earnest: the 8-site ring at half filling (a textbook
        # test system and the inner call of small solvers); latency counts.
        dict(name="hv_ring8_fp64", kind="hv", model="ring", L=8, up=4, dn=4, fp=64),
        # An ordinary one: 12 sites of a t-t' torus, unequal spin sectors that end
        # in ragged blocks, single precision as inside a mixed solve.
        dict(name="hv_torus4x3_fp32", kind="hv", model="torus4x3", L=12, up=5, dn=6, fp=32),
        # The largest: the 4x4 t-t' torus, 1.3e8 states, in single precision ...
        dict(name="hv_torus4x4_fp32", kind="hv", model="torus4x4", L=16, up=7, dn=7, fp=32),
        # ... and in double precision, as every refinement and all-FP64 solve runs it.
        dict(name="hv_torus4x4_fp64", kind="hv", model="torus4x4", L=16, up=5, dn=6, fp=64),
        # H·v over a general state set: every S_z of the 12-site ring at 12 particles,
        # which the spin-factored index cannot hold.
        dict(name="set_hv_ring12_fp32", kind="set_hv", model="ring", L=12, N=12, fp=32),
        # H·v of a list of operator products: the momentum-space ring in one
        # total-momentum sector (two-body terms in the hundreds).
        dict(name="term_hv_momentum12_fp64", kind="term_hv", L=12, up=6, dn=6, K=0, fp=64),
        # A small ground-state solve to full accuracy: double precision with
        # re-orthogonalisation, many short steps.
        dict(name="lanczos_ring8_fp64", kind="lanczos", model="ring", L=8, up=4, dn=4, iters=100, prec="fp64",
             reorth=True, graph=False),
        # An ordinary ground-state solve: 14-site ring, 1.2e7 states, mixed precision
        # with the double-precision refinement.
        dict(name="lanczos_ring14_mixed", kind="lanczos", model="ring", L=14, up=7, dn=7, iters=80, prec="mixed",
             reorth=False, graph=True),
        # Impurity solving: every particle-number sector of many small Anderson models.
        dict(name="batch_siam256", kind="batch", models=256, iters=150),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


_MODELS = [("ring", L) for L in range(6, 19)] + [("chain", L) for L in range(6, 19)] + \
          [("torus3x2", 6), ("torus4x2", 8), ("torus3x3", 9), ("torus4x3", 12), ("torus4x4", 16)] + \
          [("siam", L) for L in range(6, 13)]


def _sector(rng, lo, hi):
    """A model and particle numbers whose sector has about exp(uniform(log)) states."""
    want = math.log(_log(rng, lo, hi))
    fits = []
    while not fits:
        model, L = rng.choice(_MODELS)
        fits = [(u, d) for u in range(1, L) for d in range(1, L)
                if abs(math.log(math.comb(L, u) * math.comb(L, d)) - want) < 0.35
                and math.comb(L, u) * math.comb(L, d) <= hi]
    u, d = rng.choice(fits)
    return dict(model=model, L=L, up=u, dn=d)


def draw(rng):
    kind = rng.choice(["comb_rank", "comb_unrank", "trie_rank", "hv", "hv", "hv", "set_hv", "term_hv", "lanczos",
                       "batch"])
    if kind in ("comb_rank", "comb_unrank"):
        M = rng.randint(16, 62)
        N = rng.randint(M // 5 + 1, M - M // 5 - 1)
        n = int(_log(rng, 1 << 10, 1 << (26 if kind == "comb_rank" else 24)))
        c = dict(kind=kind, M=M, N=N, n=n, bits=64 if math.comb(M, N) > 1 << 31 else rng.choice([32, 64]))
        return dict(c, check=rng.randint(0, 1)) if kind == "comb_rank" else c
    if kind == "trie_rank":
        width = rng.randint(24, 48)
        return dict(kind=kind, width=width, members=int(_log(rng, 1 << 12, 1 << 21)), n=int(_log(rng, 1 << 10, 1 << 24)),
                    bits=rng.choice([32, 64]), check=rng.randint(0, 1), msb=rng.random() < 0.5)
    if kind == "hv":
        fp = rng.choice([32, 64])
        return dict(kind=kind, **_sector(rng, 1e3, LARGEST_HV if fp == 32 else 3.4e7), fp=fp)
    if kind == "set_hv":
        L = rng.randint(7, 12)
        N = rng.randint(max(3, L // 2), min(2 * L - 3, L + 4))
        return dict(kind=kind, model=rng.choice(["ring", "chain"]), L=L, N=N, fp=rng.choice([32, 64]))
    if kind == "term_hv":
        L = rng.randint(6, 12)
        up, dn = rng.randint(2, L - 2), rng.randint(2, L - 2)
        return dict(kind=kind, L=L, up=up, dn=dn, K=rng.randint(0, L - 1), fp=rng.choice([32, 64]))
    if kind == "lanczos":
        reorth = rng.random() < 0.4
        prec = rng.choice(["fp64", "mixed"])
        return dict(kind=kind, **_sector(rng, 1e3, 2e4 if reorth else 4e6), iters=rng.randint(30, 100), prec=prec,
                    reorth=reorth, graph=not reorth and rng.random() < 0.5)
    return dict(kind=kind, models=int(_log(rng, 2, 200)), iters=rng.randint(80, 200))


# ------------------------------------------------- models (one-body matrix, U)

def _bonds(model, L):
    """[(site, site, amplitude)] of h = -t, -t'."""
    if model in ("ring", "chain"):
        return [(i, i + 1, -1.0) for i in range(L - 1)] + ([(L - 1, 0, -1.0)] if model == "ring" else [])
    w, v = (int(t) for t in model[5:].split("x"))
    at = lambda x, y: (y % v) * w + x % w
    out = []
    for x, y in itertools.product(range(w), range(v)):
        out += [(at(x, y), at(x + 1, y), -1.0), (at(x, y), at(x, y + 1), -1.0),
                (at(x, y), at(x + 1, y + 1), 0.3), (at(x, y), at(x + 1, y - 1), 0.3)]
    return [b for b in out if b[0] != b[1]]


def _anderson(L, rng, U=4.0):
    """Impurity on site 0, bath energies in [-2, 2), hybridisations in [0, 1)."""
    h = np.zeros((L, L))
    h[0, 0] = -U / 2
    h[np.arange(1, L), np.arange(1, L)] = rng.uniform(-2, 2, L - 1)
    h[0, 1:] = h[1:, 0] = rng.uniform(0, 1, L - 1)
    return h, np.array([U] + [0.0] * (L - 1))


def _model(c, seed):
    L = c["L"]
    if c["model"] == "siam":
        return _anderson(L, np.random.default_rng(seed))
    h = np.zeros((L, L))
    for a, b, t in _bonds(c["model"], L):
        h[a, b] += t
        h[b, a] += t
    # one point of a scan over the interaction
    U = (8.0 if c["model"].startswith("torus") else 4.0) * np.random.default_rng(seed).uniform(0.75, 1.25)
    return h, np.full(L, U)


def _batch_models(c, seed):
    # 5 to 7 bath sites, uneven; the sizes belong to the case, the values to the seed
    sizes = np.random.default_rng(c["models"]).integers(6, 9, c["models"])
    rng = np.random.default_rng(seed)
    return [_anderson(int(L), rng) for L in sizes]


def _momentum_terms(L, t=1.0, U=4.0):
    """(coefficient, [operator codes, left to right]); code = 2 * orbital + creator,
    orbital m for momentum m spin down, L + m for spin up."""
    out = [(-2 * t * math.cos(2 * math.pi * m / L), [2 * (o + m) + 1, 2 * (o + m)]) for m in range(L) for o in (0, L)]
    for m, p, q in itertools.product(range(L), repeat=3):
        out.append((U / L, [2 * (L + (m + q) % L) + 1, 2 * ((p - q) % L) + 1, 2 * p, 2 * (L + m)]))
    return out


@functools.lru_cache(maxsize=64)
def _patterns(L, N):
    """All L-bit patterns with N bits set, in increasing order (int64)."""
    a = np.arange(1 << L, dtype=np.int64)
    n = np.zeros(1 << L, dtype=np.int8)
    for b in range(L):
        n += ((a >> b) & 1).astype(np.int8)
    return a[n == N]


def _states(c):
    if c["kind"] == "set_hv":
        return _patterns(2 * c["L"], c["N"])
    L = c["L"]
    momentum = lambda a: sum(m * ((a >> m) & 1) for m in range(L))
    up, dn = _patterns(L, c["up"]), _patterns(L, c["dn"])
    keep = (momentum(up)[:, None] + momentum(dn)[None, :]) % L == c["K"]
    return ((up[:, None] << L) | dn[None, :])[keep]


def _dim(c):
    return math.comb(c["L"], c["up"]) * math.comb(c["L"], c["dn"])


# ------------------------------------------------------------ inputs and passes

def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed(seed * 16 + k)


def _vector(n, seed, dtype):
    """uniform [-1, 1): the start vector of a solve."""
    return torch.empty(n, dtype=dtype, device="cuda").uniform_(-1, 1, generator=_gen(seed))


def _rank_inputs(c, seed):
    """(indices, their patterns) of a combination sector."""
    M, N = c["M"], c["N"]
    r = torch.randint(0, math.comb(M, N), (c["n"],), dtype=torch.int64, device="cuda", generator=_gen(seed))
    pat = torch.empty_like(r)
    binom = torch.tensor([[min(math.comb(p, k), (1 << 63) - 1) for k in range(M + 1)] for p in range(M)],
                         dtype=torch.int64, device="cuda")
    for lo in range(0, c["n"], 1 << 24):
        rest, a = r[lo:lo + (1 << 24)].clone(), torch.zeros_like(r[lo:lo + (1 << 24)])
        k = torch.full_like(rest, N)
        for p in range(M - 1, -1, -1):
            b = binom[p][k]
            take = ((rest >= b) & (k > 0)).to(torch.int64)
            rest -= b * take
            k -= take
            a |= take << p
        pat[lo:lo + (1 << 24)] = a
    return r, pat


def _trie_inputs(c, seed):
    """(sorted members, queries): with the check one query in eight is a stranger."""
    draw_ = lambda n, k: torch.randint(0, 1 << c["width"], (n,), dtype=torch.int64, device="cuda", generator=_gen(seed, k))
    m = torch.unique(draw_(c["members"], 1))
    q = m[torch.randint(0, m.numel(), (c["n"],), device="cuda", generator=_gen(seed, 2))]
    if c["check"]:
        strangers = torch.randint(0, 8, (c["n"],), device="cuda", generator=_gen(seed, 3)) == 0
        q = torch.where(strangers, draw_(c["n"], 4), q)
    return m, q


def prepare(case, seed):
    c, kind = case, case["kind"]
    whole = {32: torch.int32, 64: torch.int64}
    real = {32: torch.float32, 64: torch.float64}
    if kind in ("comb_rank", "comb_unrank"):
        r, pat = _rank_inputs(c, seed)
        s = dict(kind=kind, h=G.gbr_comb_create(c["M"], c["N"], 8))
        if kind == "comb_rank":
            return dict(s, pat=pat, out=torch.empty(c["n"], dtype=whole[c["bits"]], device="cuda"), check=c["check"])
        return dict(s, rank=r.to(whole[c["bits"]]), out=pat)
    if kind == "trie_rank":
        m, q = _trie_inputs(c, seed)
        h = G.gbr_trie_create(m.cpu().numpy().view(np.uint64), c["width"], 8, c["msb"])
        return dict(kind=kind, h=h, pat=q, out=torch.empty(c["n"], dtype=whole[c["bits"]], device="cuda"), check=c["check"])
    if kind == "batch":
        models = _batch_models(c, seed)
        return dict(kind=kind, models=models, iters=c["iters"],
                    start=_vector(G.gbr_batch_layout(models)[1], seed, torch.float64))
    if kind == "term_hv":
        terms = [G.gbr_term_product(ops, v) for v, ops in _momentum_terms(c["L"])]
        st = _states(c)
        h = G.gbr_termham_create(2 * c["L"], terms, st.view(np.uint64), 8)
        n, dtype = st.size, real[c["fp"]]
    elif kind == "set_hv":
        st = _states(c)
        h = G.gbr_setham_create(c["L"], *_model(c, seed), st.view(np.uint64), 8)
        n, dtype = st.size, real[c["fp"]]
    else:
        hm, U = _model(c, seed)
        h = G.gbr_ham_create(c["L"], hm, U, c["up"], c["dn"])
        n = _dim(c)
        if kind == "lanczos":
            return dict(kind=kind, h=h, v0=_vector(n, seed, torch.float64), c=c,
                        prec=G.GBR_PREC_FP64 if c["prec"] == "fp64" else G.GBR_PREC_MIXED)
        dtype = real[c["fp"]]
    x = _vector(n, seed, dtype)
    return dict(kind=kind, h=h, x=x, y=torch.empty_like(x))


def run(state):
    s = state
    kind = s["kind"]
    if kind == "comb_rank":
        return G.gbr_comb_rank(s["h"], s["pat"], s["out"], check=s["check"])
    if kind == "comb_unrank":
        return G.gbr_comb_unrank(s["h"], s["rank"], s["out"])
    if kind == "trie_rank":
        return G.gbr_trie_rank(s["h"], s["pat"], s["out"], check=s["check"])
    if kind == "hv":
        return G.gbr_hv(s["h"], s["x"], s["y"])
    if kind == "set_hv":
        return G.gbr_setham_hv(s["h"], s["x"], s["y"], check=1)
    if kind == "term_hv":
        return G.gbr_termham_hv(s["h"], s["x"], s["y"], check=1)
    if kind == "lanczos":
        c = s["c"]
        r = G.gbr_lanczos(s["h"], s["v0"], c["iters"], reorth=c["reorth"], prec=s["prec"], refine=True,
                          use_graph=c["graph"])
        # without re-orthogonalisation the coefficients past convergence are
        # decided by rounding, so a program reads the energies alone
        keys = ("E0", "E_ritz", "alpha", "beta") if c["reorth"] else ("E0", "E_ritz")
        return {k: np.atleast_1d(r[k]) for k in keys}
    r = G.gbr_batch_solve(s["models"], s["start"], s["iters"])
    return {k: r[k] for k in ("E0", "sector_E", "arg")}


# --------------------------------------------------- bytes, operations, limits

def _hops(h, L, N):
    """Valid hops of all L-bit patterns with N particles."""
    return int(np.count_nonzero(h - np.diag(np.diag(h)))) * math.comb(L - 2, N - 1)


def _elements(c):
    """Matrix elements of one H·v of a spin-factored sector."""
    h, _ = _model(c, 0)
    du, dd = math.comb(c["L"], c["up"]), math.comb(c["L"], c["dn"])
    return du * dd + _hops(h, c["L"], c["up"]) * dd + _hops(h, c["L"], c["dn"]) * du


def work(case):
    c, kind = case, case["kind"]
    if kind in ("comb_rank", "comb_unrank"):
        return {"bytes": c["n"] * (8 + c["bits"] // 8), "flops": 0}
    if kind == "trie_rank":
        # patterns in, ranks out, and the members themselves once
        return {"bytes": c["n"] * (8 + c["bits"] // 8) + 8 * c["members"], "flops": 0}
    if kind == "hv":
        return {"bytes": 2 * _dim(c) * c["fp"] // 8, "flops": 2 * _elements(c)}
    if kind == "set_hv":
        h, _ = _model(c, 0)
        n = math.comb(2 * c["L"], c["N"])
        bonds = int(np.count_nonzero(h)) * 2 * math.comb(2 * c["L"] - 2, c["N"] - 1)
        return {"bytes": n * (8 + 2 * c["fp"] // 8), "flops": 2 * (n + bonds)}
    if kind == "term_hv":
        n = _dim(c) // c["L"]
        # diagonal, and every pair of an up and a down particle scattering by q
        return {"bytes": n * (8 + 2 * c["fp"] // 8), "flops": 2 * n * (2 * c["L"] + c["up"] * c["dn"] * (c["L"] - max(c["up"], c["dn"])))}
    if kind == "lanczos":
        b = 8 if c["prec"] == "fp64" else 4
        n, k = _dim(c), c["iters"]
        reorth = 2 * k * k * n if c["reorth"] else 0
        return {"bytes": 8 * n + 3 * k * b * n, "flops": 2 * k * _elements(c) + 10 * k * n + 2 * reorth}
    # about 30 steps a sector, each an H·v of 2 (1 + 2 bath) elements a state
    n = c["models"] * (4 ** 6 + 4 ** 7 + 4 ** 8) // 3
    return {"bytes": 8 * n, "flops": 30 * n * 40}


def tolerance(case):
    c, kind = case, case["kind"]
    if kind in ("comb_rank", "comb_unrank", "trie_rank"):
        return "exact"
    # each figure is about four times the largest error seen against exact()
    if kind in ("hv", "set_hv", "term_hv"):
        # tens to hundreds of products a state, each and their sum rounded at 2^-24 or 2^-53
        if c["fp"] == 64:
            return {"rel": 2e-15, "max": 2e-14}
        return {"rel": 1.2e-6 if kind == "term_hv" else 4e-7, "max": 1e-5}
    if kind == "lanczos":
        if c["prec"] == "fp64":
            return {"rel": 1e-12, "max": 1e-10}
        # single-precision vectors move the unrefined energy and the coefficients by their rounding
        return {"rel": 1e-6, "max": 1e-5} if c["reorth"] else {"rel": 1.5e-7}
    # energies come from vectors converged to 1e-6; equal minima of two sectors are ties
    return {"rel": 1e-11, "max": 1e-9, "differ": 0.01}


# ------------------------------------------------------- the outputs in 64 bits

def _parity(v):
    for s in (32, 16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return v & 1


def _between(p, q):
    lo, hi = min(p, q), max(p, q)
    return ((1 << hi) - 1) & ~((1 << (lo + 1)) - 1)


def _spin_matrix(h, L, N):
    """One spin's hopping as a sparse CSR matrix (FP64, on the GPU), its
    one-body diagonal and its patterns."""
    st = _patterns(L, N)
    rows, cols, vals = [], [], []
    for p, q in itertools.permutations(range(L), 2):
        if h[p, q]:
            ok = np.nonzero(((st >> p) & 1 == 1) & ((st >> q) & 1 == 0))[0]
            to = st[ok] ^ ((1 << p) | (1 << q))
            rows.append(ok)
            cols.append(np.searchsorted(st, to))
            vals.append(h[p, q] * (1 - 2 * _parity(st[ok] & _between(p, q))))
    cat = lambda v, t: torch.from_numpy(np.concatenate(v).astype(t)).cuda() if v else torch.zeros(0, device="cuda")
    m = torch.sparse_coo_tensor(torch.stack([cat(rows, np.int64), cat(cols, np.int64)]), cat(vals, np.float64),
                                (st.size, st.size)).to_sparse_csr()
    diag = sum(h[p, p] * ((st >> p) & 1) for p in range(L)).astype(np.float64)
    return m, torch.from_numpy(diag).cuda(), torch.from_numpy(st).cuda()


def _sector_op(h, U, L, up, dn):
    """x -> H x on the (up, dn) sector, FP64."""
    mu, du, su = _spin_matrix(h, L, up)
    md, dd, sd = _spin_matrix(h, L, dn)

    def apply(x):
        X = x.double().view(su.numel(), sd.numel())
        Y = torch.empty_like(X)
        for lo in range(0, su.numel(), 512):
            both = su[lo:lo + 512, None] & sd[None, :]
            d = du[lo:lo + 512, None] + dd[None, :]
            for p in range(L):
                if U[p]:
                    d = d + U[p] * ((both >> p) & 1).double()
            Y[lo:lo + 512] = d * X[lo:lo + 512] + (md @ X[lo:lo + 512].T.contiguous()).T
        for lo in range(0, sd.numel(), 2048):
            Y[:, lo:lo + 2048] += mu @ X[:, lo:lo + 2048].contiguous()
        return Y.view(-1)

    return apply


def _lanczos64(apply, v, iters):
    """alpha, beta of the recurrence with two Gram-Schmidt passes."""
    V = [v.double() / torch.linalg.vector_norm(v.double())]
    a, b = [], []
    for k in range(min(iters, v.numel())):
        w = apply(V[k])
        if k:
            w = w - b[-1] * V[k - 1]
        a.append(float(torch.dot(w, V[k])))
        w = w - a[-1] * V[k]
        for _ in range(2):
            for u in V:
                w = w - torch.dot(w, u) * u
        n = float(torch.linalg.vector_norm(w))
        if k + 1 == min(iters, v.numel()) or n <= 1e-13 * max(max(map(abs, a)), max(b, default=0.0)):
            break
        b.append(n)
        V.append(w / n)
    return np.array(a), np.array(b)


def _lowest(a, b):
    return float(np.linalg.eigvalsh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))[0])


def _exact_set(c, seed):
    h, U = _model(c, seed)
    L = c["L"]
    st = torch.from_numpy(_states(c)).cuda()
    x = _vector(st.numel(), seed, torch.float32 if c["fp"] == 32 else torch.float64).double()
    ad, au = st & ((1 << L) - 1), st >> L
    d = torch.zeros_like(x)
    for p in range(L):
        d += h[p, p] * (((ad >> p) & 1) + ((au >> p) & 1)).double() + U[p] * (((ad & au) >> p) & 1).double()
    y = d * x
    for p, q in itertools.permutations(range(L), 2):
        for off, a in ((0, ad), (L, au)) if h[p, q] else ():
            ok = torch.nonzero(((a >> p) & 1 == 1) & ((a >> q) & 1 == 0)).view(-1)
            to = st[ok] ^ (((1 << p) | (1 << q)) << off)
            j = torch.searchsorted(st, to).clamp_max(st.numel() - 1)
            s = h[p, q] * (1 - 2 * _parity(a[ok] & _between(p, q))).double() * (st[j] == to)
            y[ok] += s * x[j]
    return y


def _exact_terms(c, seed):
    st = torch.from_numpy(_states(c)).cuda()
    x = _vector(st.numel(), seed, torch.float32 if c["fp"] == 32 else torch.float64).double()
    y = torch.zeros_like(x)
    for v, ops in _momentum_terms(c["L"]):
        a, ok, sign = st.clone(), torch.ones_like(st, dtype=torch.bool), torch.ones_like(x)
        for code in reversed(ops):
            o = code >> 1
            ok &= ((a >> o) & 1) == (0 if code & 1 else 1)
            sign *= 1 - 2 * _parity(a & ((1 << o) - 1)).double()
            a = a ^ (1 << o)
        j = torch.searchsorted(st, a).clamp_max(st.numel() - 1)
        ok &= st[j] == a
        y.index_add_(0, j[ok], (v * sign * x)[ok])
    return y


def _exact_batch(c, seed):
    E, first, arg = [], [], []
    for h, U in _batch_models(c, seed):
        L = h.shape[0]
        e = {}
        for u, d in itertools.product(range(L + 1), repeat=2):
            if u > d:
                e[u, d] = e[d, u]           # no field: the sectors mirror each other
                continue
            op = _sector_op(h, U, L, u, d)
            n = math.comb(L, u) * math.comb(L, d)
            g = torch.empty(n, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=_gen(seed, 5))
            e[u, d] = _lowest(*_lanczos64(op, g, 110))
        E += [e[u, d] for u, d in itertools.product(range(L + 1), repeat=2)]
        first.append(min(e.values()))
        best = min(k for k in ((u + d, u, d) for u, d in e) if e[k[1], k[2]] <= first[-1] + 1e-10 * max(1.0, abs(first[-1])))
        arg.append(best[1:])
    return {"E0": np.array(first), "sector_E": np.array(E), "arg": np.array(arg, dtype=np.int32)}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("comb_rank", "comb_unrank"):
        r, pat = _rank_inputs(c, seed)
        return pat if kind == "comb_unrank" else r.to(torch.int32 if c["bits"] == 32 else torch.int64)
    if kind == "trie_rank":
        m, q = _trie_inputs(c, seed)
        j = torch.searchsorted(m, q).clamp_max(m.numel() - 1)
        return torch.where(m[j] == q, j, -1).to(torch.int32 if c["bits"] == 32 else torch.int64)
    if kind == "hv":
        x = _vector(_dim(c), seed, torch.float32 if c["fp"] == 32 else torch.float64)
        return _sector_op(*_model(c, seed), c["L"], c["up"], c["dn"])(x)
    if kind == "set_hv":
        return _exact_set(c, seed)
    if kind == "term_hv":
        return _exact_terms(c, seed)
    if kind == "lanczos":
        a, b = _lanczos64(_sector_op(*_model(c, seed), c["L"], c["up"], c["dn"]), _vector(_dim(c), seed, torch.float64),
                          c["iters"])
        E = np.array([_lowest(a, b)])
        return {"E0": E, "E_ritz": E, "alpha": a, "beta": b} if c["reorth"] else {"E0": E, "E_ritz": E}
    return _exact_batch(c, seed) if c["models"] <= 3 else None
