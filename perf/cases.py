"""The work a user of this framework has it do, as cases that can be timed.

A case names a system recipe (the generators of ``mbe_synth``), an entry point
and its sizes; ``prepare`` makes what a user's program holds before the call,
``run`` is one call through the public entry points, ``exact`` gives the same
outputs in 64 bits from a plain determinant-space solver written here.

Kinds:
  sigma   mbe_sigma_noalloc: one FP64 sigma vector on the caller's device
          buffers, the building block of a user's own eigensolver
  solve   mbe_solve_tuples: the CASCI energies of a set of tuples of one order
  expand  MBE.run: a whole screened expansion, order by order
  grad    autograd.mbe_energy and its backward: the energy and its gradient
          with respect to the integrals
"""
import itertools
import math

import numpy as np
import torch

from paper_1905_02786_gb300 import _binding as B
from paper_1905_02786_gb300 import autograd

# integral recipes of mbe_synth's workloads: the water-shaped one (well
# separated virtuals) and the hydrogen-chain-shaped one (near-degenerate)
RECIPES = {"dz": dict(eps_occ=(-1.5, -0.4), eps_vir=(0.05, 3.0), mean_pppp=0.5),
           "chain": dict(eps_occ=(-0.6, -0.3), eps_vir=(0.0, 1.5), mean_pppp=0.6)}
SPIN_SHIFT = 0.5                                # the library's default lambda
TIGHT = dict(conv_tol_r=1e-11, conv_tol_e=1e-14)
# sigma vectors of one converged CASCI, about what the repository's workloads
# take (40 on the water-shaped system)
SIGMAS = 40


def listed():
    return [
        # one FP64 sigma vector of a small active space: a call a user's own
        # iteration makes thousands of times (latency and launches)
        dict(name="sigma_6e8o", kind="sigma", recipe="dz", norb=12, nel=6, two_sz=0,
             lo=0, hi=8),
        # the largest closed-shell space this entry point takes
        dict(name="sigma_8e9o", kind="sigma", recipe="dz", norb=14, nel=8, two_sz=0,
             lo=0, hi=9),
        # order 1 of the 8e/23o workload at the library's defaults (FP64): 17
        # small CASCIs in two uneven bins, 6e/7o and 8e/7o
        dict(name="fp64_order1_8e23o", kind="solve", recipe="dz", norb=23, nel=8, two_sz=0,
             lo=1, hi=7, order=1, count=17, holes="any", precision="fp64"),
        # order 3 of the same workload, FP64: 6e/9o and 8e/9o
        dict(name="fp64_order3_8e23o", kind="solve", recipe="dz", norb=23, nel=8, two_sz=0,
             lo=1, hi=7, order=3, count=45, holes="any", precision="fp64"),
        # FP64 energies of a few larger CASCIs (8e/11o, 108,900 determinants):
        # what a user checks the mixed path with
        dict(name="fp64_8e11o", kind="solve", recipe="dz", norb=23, nel=8, two_sz=0,
             lo=1, hi=7, order=5, count=3, holes="in", precision="fp64"),
        # high-spin reference (a doublet): different alpha and beta strings
        dict(name="fp64_doublet_7e9o", kind="solve", recipe="dz", norb=14, nel=7, two_sz=1,
             lo=1, hi=6, order=3, count=24, holes="any", precision="fp64"),
        # energy and integral gradient of the differentiation workload's
        # system, unscreened to order 3, through torch.autograd
        dict(name="grad_8e20o_order3", kind="grad", recipe="dz", norb=20, nel=8, two_sz=0,
             lo=2, hi=6, order=3),
        # the benchmark's expansion (mixed precision) up to order 3: tuple
        # generation, uneven bins, increments, screening
        dict(name="expand_8e23o_order3", kind="expand", recipe="dz", norb=23, nel=8, two_sz=0,
             lo=1, hi=7, order=3, thr=1e-6, precision="mixed"),
        # the benchmark's most frequent bin, order 6 without the inactive
        # occupied orbital: 6e/12o, 48,400 determinants each
        dict(name="mixed_6e12o", kind="solve", recipe="dz", norb=23, nel=8, two_sz=0,
             lo=1, hi=7, order=6, count=96, holes="out", precision="mixed"),
        # its largest bin: 8e/12o, 245,025 determinants each
        dict(name="mixed_8e12o", kind="solve", recipe="dz", norb=23, nel=8, two_sz=0,
             lo=1, hi=7, order=6, count=64, holes="in", precision="mixed"),
        # near-degenerate chain, order 2: 10e/12o, 627,264 determinants each
        dict(name="mixed_chain_10e12o", kind="solve", recipe="chain", norb=32, nel=10, two_sz=0,
             lo=0, hi=10, order=2, count=8, holes="any", precision="mixed"),
        # order 3 of the chain: 10e/13o, 1,656,369 determinants
        dict(name="mixed_chain_10e13o", kind="solve", recipe="chain", norb=32, nel=10, two_sz=0,
             lo=0, hi=10, order=3, count=1, holes="any", precision="mixed"),
    ]


def _loguni(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ndet(n, na, nb):
    return math.comb(n, na) * math.comb(n, nb)


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "fp64", "fp64", "open", "grad", "expand", "mixed",
                       "mixed", "mixed", "chain"])
    if kind == "sigma":
        n = rng.randint(5, 9)
        occ = rng.randint(2, 4)
        norb = rng.randint(n + 1, 20)
        lo = rng.randint(0, min(1, norb - n))
        return dict(kind="sigma", recipe=rng.choice(["dz", "chain"]), norb=norb, nel=2 * (occ + lo),
                    two_sz=0, lo=lo, hi=lo + n)
    if kind == "grad":
        return dict(kind="grad", recipe="dz", norb=rng.randint(9, 20), nel=8, two_sz=0,
                    lo=2, hi=6, order=rng.randint(1, 3))
    if kind == "expand":
        return dict(kind="expand", recipe="dz", norb=rng.randint(12, 23), nel=8, two_sz=0,
                    lo=1, hi=7, order=rng.randint(1, 3), thr=float("%.2e" % 10 ** rng.uniform(-7, -5)),
                    precision="mixed")
    if kind == "open":
        two_sz = rng.randint(1, 2)
        return dict(kind="solve", recipe="dz", norb=rng.randint(10, 20), nel=6 + two_sz,
                    two_sz=two_sz, lo=1, hi=6, order=rng.randint(1, 3), count=_loguni(rng, 1, 48),
                    holes="any", precision="fp64")
    if kind == "fp64":
        order = rng.randint(1, 5)
        most = {1: 17, 2: 64, 3: 64, 4: 12, 5: 3}[order]
        return dict(kind="solve", recipe="dz", norb=rng.randint(16, 23), nel=8, two_sz=0, lo=1,
                    hi=7, order=order, count=_loguni(rng, 1, most),
                    holes=rng.choice(["any", "in", "out"]) if order > 1 else "any",
                    precision="fp64")
    if kind == "mixed":
        order = rng.randint(2, 6)
        return dict(kind="solve", recipe="dz", norb=rng.randint(16, 23), nel=8, two_sz=0, lo=1,
                    hi=7, order=order, count=_loguni(rng, 2, 64),
                    holes=rng.choice(["any", "in", "out"]), precision="mixed")
    order = rng.randint(1, 2)
    return dict(kind="solve", recipe="chain", norb=rng.randint(16, 40), nel=10, two_sz=0, lo=0,
                hi=10, order=order, count=_loguni(rng, 1, 6), holes="any", precision="mixed")


# ------------------------------------------------------------------ inputs
def _spaces(case):
    ref = list(range(case["lo"], case["hi"]))
    return ref, [o for o in range(case["norb"]) if o not in ref]


def _occ(case):
    nb = (case["nel"] - case["two_sz"]) // 2
    return nb + case["two_sz"], nb


def _integrals(case, seed):
    """The recipe of mbe_synth.gen_integrals, drawn from this case's seed."""
    import mbe_synth as ms
    return ms.gen_integrals(case["norb"], _occ(case)[1], seed, **RECIPES[case["recipe"]])[:2]


def _tuples(case, seed):
    """`count` distinct tuples of the expansion orbitals (all of them if there
    are no more); holes "in" / "out": with / without the lowest expansion
    orbital (an inactive occupied one, where there is one)."""
    _, exp = _spaces(case)
    k = case["order"]
    rest = exp if case["holes"] == "any" else exp[1:]
    kk = k - 1 if case["holes"] == "in" else k
    fix = (exp[0],) if case["holes"] == "in" else ()
    total = math.comb(len(rest), kk)
    if total <= case["count"]:
        return [fix + t for t in itertools.combinations(rest, kk)]
    rng, seen = np.random.default_rng(seed), set()
    while len(seen) < case["count"]:
        seen.add(tuple(sorted(int(x) for x in rng.choice(rest, size=kk, replace=False))))
    return [fix + t for t in sorted(seen)]


def _options(case):
    return dict(precision=B.MBE_MIXED_BF16X3, max_batch=4096) if case.get("precision") == "mixed" else {}


def prepare(case, seed):
    B.load_library()
    h, eri = _integrals(case, seed)
    ref, exp = _spaces(case)
    if case["kind"] == "grad":
        t = dict(dtype=torch.float64, device="cuda")
        return dict(kind="grad", h=torch.tensor(h, **t).requires_grad_(),
                    eri=torch.tensor(eri, **t).requires_grad_(), nel=case["nel"], ref=ref,
                    exp=exp, order=case["order"])
    m = B.MBE(0, **_options(case))
    m.load(h, eri, case["nel"], two_sz=case["two_sz"])
    s = dict(kind=case["kind"], m=m, ref=ref, exp=exp)
    if case["kind"] == "sigma":
        na, _ = _occ(case)
        nstr = math.comb(len(ref), sum(o < na for o in ref))
        s["c"] = torch.tensor(_vector(nstr, seed), device="cuda")
        s["sigma"] = torch.empty_like(s["c"])
    elif case["kind"] == "solve":
        B.mbe_set_reference(m.ctx, ref, exp)
        s["tuples"], s["order"] = np.array(_tuples(case, seed), dtype=np.int32), case["order"]
    else:
        s["order"], s["thr"] = case["order"], case["thr"]
    return s


def _vector(nstr, seed):
    """A normalised CI vector, one determinant dominating as in a converged
    state, not symmetric (the entry point takes any)."""
    rng = np.random.default_rng(seed + 1)
    c = 0.2 * rng.standard_normal((nstr, nstr)) / nstr
    c[0, 0] += 1.0
    return c / np.linalg.norm(c)


def run(state):
    kind = state["kind"]
    if kind == "grad":
        e = autograd.mbe_energy(state["h"], state["eri"], state["nel"], state["ref"], state["exp"],
                                state["order"], 0.0, 0, **TIGHT)
        dh, deri = torch.autograd.grad(e, (state["h"], state["eri"]))
        return {"energy": e.detach(), "dh": dh, "deri": deri}
    m = state["m"]
    if kind == "sigma":
        B.mbe_sigma_noalloc(m.ctx, state["ref"], state["c"], state["sigma"], want_core=False)
        return {"sigma": state["sigma"]}
    if kind == "solve":
        eps, status = B.mbe_solve_tuples(m.ctx, state["tuples"], state["order"], allow_noconv=True)
        return {"eps": eps, "status": status}
    res = m.run(state["ref"], state["exp"], state["order"], state["thr"])
    o = res["orders"]
    return _expansion(res["eps_ref"], [r["E_order"] for r in o], res["total"],
                      np.concatenate([r["eps"] for r in o]), np.concatenate([r["inc"] for r in o]),
                      np.concatenate([r["keep"] for r in o]))


def _expansion(e_ref, e_order, total, eps, inc, keep):
    """Everything an expansion returns: the reference, order and total
    energies, one row (energy, increment) per tuple, the screening flags."""
    return {"energies": np.array([e_ref, *e_order, total]),
            "tuples": np.stack([eps, inc], axis=1), "keep": keep}


# ------------------------------------------------------------------ work
def _sizes(case):
    """(orbitals, alpha, beta electrons) of every CASCI of the call."""
    na, nb = _occ(case)
    ref, exp = _spaces(case)
    if case["kind"] == "sigma":
        sets = [()]
    elif case["kind"] == "solve":
        sets = _tuples(case, 0)
    else:
        sets = [t for k in range(case["order"] + 1) for t in itertools.combinations(exp, k)]
    return [(len(ref) + len(t), sum(o < na for o in itertools.chain(ref, t)),
             sum(o < nb for o in itertools.chain(ref, t))) for t in sets]


def work(case):
    """Bytes: the integrals and every CASCI's vectors (read one, write one per
    sigma vector) and the outputs; flops: the non-zero elements of the CASCI
    Hamiltonian times two per sigma vector."""
    by = fl = 0.0
    npg = case["norb"] * (case["norb"] + 1) // 2
    width = 4 if case.get("precision") == "mixed" else 8
    nsig = 1 if case["kind"] == "sigma" else SIGMAS
    sizes = _sizes(case)
    for n, a, b in sizes:
        ndet = _ndet(n, a, b)
        sa, sb = a * (n - a), b * (n - b)
        same = lambda k: math.comb(k, 2) * math.comb(n - k, 2)      # noqa: E731
        fl += 2.0 * nsig * ndet * (1 + sa + sb + sa * sb + same(a) + same(b))
        by += 2.0 * nsig * ndet * width
    if case["kind"] == "sigma":
        n = case["hi"] - case["lo"]
        by += 8.0 * (n * (n + 1) // 2) ** 2
    else:
        by += 8.0 * npg * npg * (2 if case["kind"] == "grad" else 1) + 16.0 * len(sizes)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ exact
# A determinant-space solver in plain torch, FP64, batched over the CASCIs of
# one shape: sigma = 1/2 sum_PQ g'_PQ E_P E_Q c + lambda S^2 c by index
# tables, a Davidson iteration without shortcuts.
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _strings(n, k):
    return [m for m in range(1 << n) if bin(m).count("1") == k]


def _links(n, k):
    """idx[P][I], sgn[P][I] of <I|E_pq + E_qp|J> (E_pp for p = q)."""
    s = _strings(n, k)
    rank = {m: i for i, m in enumerate(s)}
    np_ = n * (n + 1) // 2
    idx, sgn = np.zeros((np_, len(s)), dtype=np.int64), np.zeros((np_, len(s)))
    for p in range(n):
        for q in range(p + 1):
            P = p * (p + 1) // 2 + q
            for i, m in enumerate(s):
                if p == q:
                    if m >> p & 1:
                        idx[P, i], sgn[P, i] = i, 1.0
                elif (m >> p & 1) != (m >> q & 1):
                    between = m & ((1 << p) - 1) & ~((2 << q) - 1)
                    idx[P, i] = rank[m ^ (1 << p) ^ (1 << q)]
                    sgn[P, i] = -1.0 if bin(between).count("1") & 1 else 1.0
    return torch.from_numpy(idx).to(_dev()), torch.from_numpy(sgn).to(_dev())


def _occupation(n, k):
    return torch.tensor([[float(m >> p & 1) for p in range(n)] for m in _strings(n, k)],
                        dtype=torch.float64, device=_dev()).reshape(-1, n)


class _Shape:
    def __init__(self, n, a, b):
        self.n, self.a, self.b = n, a, b
        self.A, self.B = _links(n, a), _links(n, b)
        self.oa, self.ob = _occupation(n, a), _occupation(n, b)
        ms = 0.5 * (a - b)
        self.s2d = b - self.oa @ self.ob.T + ms * (ms + 1)

    def D(self, c):
        """D[t, P, Ia, Ib] = (E_P c)(Ia, Ib), both spins."""
        ia, sa = self.A
        ib, sb = self.B
        t, npr = c.shape[0], ia.shape[0]
        x = c[:, ia.reshape(-1)].reshape(t, npr, *c.shape[1:]) * sa[None, :, :, None]
        y = c[:, :, ib.reshape(-1)].reshape(t, c.shape[1], npr, c.shape[2]).transpose(1, 2)
        return x + y * sb[None, :, None, :]

    def h(self, g, c):
        D = self.D(c)
        t, npr = D.shape[:2]
        E = (g @ D.reshape(t, npr, -1)).reshape(D.shape)
        ia, sa = self.A
        ib, sb = self.B
        out = torch.zeros_like(c)
        for P in range(npr):
            out += E[:, P][:, ia[P]] * sa[P][None, :, None] + E[:, P][:, :, ib[P]] * sb[P]
        return 0.5 * out

    def s2(self, c):
        out = self.s2d * c
        (ia, sa), (ib, sb) = self.A, self.B
        for p in range(self.n):
            for q in range(p):
                P = p * (p + 1) // 2 + q
                up = (self.oa[:, p] * (1 - self.oa[:, q]), self.ob[:, q] * (1 - self.ob[:, p]))
                dn = (self.oa[:, q] * (1 - self.oa[:, p]), self.ob[:, p] * (1 - self.ob[:, q]))
                w = torch.outer(up[0] * sa[P], up[1] * sb[P]) + torch.outer(dn[0] * sa[P], dn[1] * sb[P])
                out -= w * c[:, ia[P]][:, :, ib[P]]
        return out


def _effective(h, eri, nb, nact_el, act):
    """E_core and the packed pair integrals g' (one-electron part folded in)
    of one active space; differentiable in h and eri."""
    norb, n = h.shape[0], len(act)
    core = [i for i in range(nb) if i not in act]
    pair = lambda p, q: p * (p + 1) // 2 + q if p >= q else q * (q + 1) // 2 + p    # noqa: E731
    dev = h.device
    ix = lambda v: torch.tensor(v, device=dev, dtype=torch.long)                    # noqa: E731
    ecore = h.new_zeros(())
    if core:
        ecore = 2 * h[ix(core), ix(core)].sum()
        ii = ix([pair(i, i) for i in core])
        ecore = ecore + 2 * eri[ii][:, ii].sum()
        ij = ix([pair(i, j) for i in core for j in core])
        ecore = ecore - eri[ij, ij].sum()
    a = ix(act)
    he = h[a][:, a]
    pq = ix([[pair(p, q) for q in act] for p in act])
    for i in core:
        pi = ix([pair(p, i) for p in act])
        he = he + 2 * eri[pq, pair(i, i)] - eri[pi][:, pi]
    hp = he
    for r in act:
        pr = ix([pair(p, r) for p in act])
        hp = hp - 0.5 * eri[pr][:, pr]
    pk = [(p, q) for p in range(n) for q in range(p + 1)]
    P = ix([pair(act[p], act[q]) for p, q in pk])
    hpk = hp[ix([p for p, _ in pk]), ix([q for _, q in pk])]
    d = torch.tensor([1.0 if p == q else 0.0 for p, q in pk], dtype=h.dtype, device=dev)
    g = eri[P][:, P]
    if nact_el:
        g = g + (torch.outer(hpk, d) + torch.outer(d, hpk)) / nact_el
    return ecore, g


def _lowest(sh, g, closed):
    """Lowest state of H + lambda S^2 (alpha-beta symmetric for a closed
    shell) of a batch: (E - lambda <S^2>, vectors)."""
    t, na, nb = g.shape[0], sh.oa.shape[0], sh.ob.shape[0]
    n = na * nb
    occ = sh.oa[:, None, :] + sh.ob[None, :, :]
    pp = torch.tensor([p * (p + 1) // 2 + p for p in range(sh.n)], device=g.device)
    off = torch.ones(g.shape[1], dtype=g.dtype, device=g.device).index_fill(0, pp, 0.0)
    exch = off * torch.diagonal(g, dim1=1, dim2=2)
    hd = 0.5 * (torch.einsum("abp,tpq,abq->tab", occ, g[:, pp][:, :, pp], occ)
                + (exch @ sh.A[1].abs())[:, :, None] + (exch @ sh.B[1].abs())[:, None, :])
    hd = hd + SPIN_SHIFT * sh.s2d
    op = lambda c: sh.h(g, c) + SPIN_SHIFT * sh.s2(c)                               # noqa: E731
    sym = (lambda c: 0.5 * (c + c.transpose(1, 2))) if closed else (lambda c: c)
    dot = lambda x, y: (x * y).sum((1, 2))                                         # noqa: E731
    c = torch.zeros(t, n, dtype=torch.float64, device=g.device)
    c[torch.arange(t), hd.reshape(t, -1).argmin(1)] = 1.0
    c = sym(c.reshape(t, na, nb))
    V, W = [], []
    m_max, x = 40, None
    for _ in range(300):
        # a correction inside the subspace (its CASCI has converged) becomes 0
        for tiny in (1e-300, 1e-7, 0.5):
            for v in V:
                c = c - dot(v, c)[:, None, None] * v
            nrm = dot(c, c).sqrt()[:, None, None]
            c = torch.where(nrm > tiny, c / nrm.clamp_min(1e-300), 0 * c)
        V.append(c)
        W.append(op(c))
        S = torch.stack(V, 1).flatten(2) @ torch.stack(W, 1).flatten(2).transpose(1, 2)
        # a vector that vanished keeps a harmless high diagonal
        S = 0.5 * (S + S.transpose(1, 2))
        dead = torch.stack([dot(v, v) < 0.5 for v in V], 1)
        S = S + torch.diag_embed(dead.to(S.dtype) * 1e6)
        ev, ec = torch.linalg.eigh(S)
        y = ec[:, :, 0]
        x = sum(y[:, i, None, None] * V[i] for i in range(len(V)))
        ax = sum(y[:, i, None, None] * W[i] for i in range(len(V)))
        r = ax - ev[:, 0, None, None] * x
        if float(dot(r, r).sqrt().max()) < 1e-12 * max(1.0, float(ev[:, 0].abs().max())):
            break
        if len(V) >= m_max:
            keep = 6
            V, W = ([sum(ec[:, i, j, None, None] * X[i] for i in range(len(X))) for j in range(keep)]
                    for X in (V, W))
        den = ev[:, 0, None, None] - hd
        den = torch.where(den.abs() < 1e-2, torch.full_like(den, -1e-2), den)
        c = sym(r / den)
    e = dot(x, op(x)) / dot(x, x)
    return e - SPIN_SHIFT * dot(x, sh.s2(x)) / dot(x, x), x / dot(x, x).sqrt()[:, None, None]


def _casci(case, h, eri, sets):
    """{tuple: (energy, vector, (n, a, b))} of every tuple in `sets`."""
    na, nb = _occ(case)
    ref, _ = _spaces(case)
    bins, out = {}, {}
    for t in sets:
        act = sorted(ref + list(t))
        key = (len(act), sum(o < na for o in act), sum(o < nb for o in act))
        bins.setdefault(key, []).append((tuple(t), act))
    for key, jobs in bins.items():
        sh = _Shape(*key)
        n, a, b = key
        step = max(1, int(2e9 / (8.0 * _ndet(n, a, b) * (n * (n + 1) // 2))))
        for j in range(0, len(jobs), step):
            part = jobs[j:j + step]
            eff = [_effective(h, eri, nb, a + b, act) for _, act in part]
            e, x = _lowest(sh, torch.stack([g for _, g in eff]), a == b)
            for i, (t, _) in enumerate(part):
                out[t] = (float(e[i] + eff[i][0]), x[i], key)
    return out


def _increments(eps, e_ref, tuples_by_order):
    inc = {}
    for tuples in tuples_by_order:
        for t in tuples:
            low = (inc[s] for k in range(1, len(t)) for s in itertools.combinations(t, k))
            inc[t] = eps[t] - e_ref - math.fsum(low)
    return inc


def _screened(case, h, eri):
    """Orders of the screened expansion: ([tuples per order], eps, inc, e_ref)."""
    _, exp = _spaces(case)
    e_ref = _casci(case, h, eri, [()])[()][0]
    orders, eps, inc = [], {}, {}
    for k in range(1, case["order"] + 1):
        if k == 1:
            tuples = [(o,) for o in exp]
        else:
            last = set(orders[-1])
            cand = sorted({t + (o,) for t in last for o in exp if o > t[-1]})
            subs = {t: list(itertools.combinations(t, k - 1)) for t in cand}
            tuples = [t for t in cand if all(s in last for s in subs[t])
                      and any(abs(inc[s]) >= case["thr"] for s in subs[t])]
        if not tuples:
            break
        orders.append(tuples)
        eps.update({t: v[0] for t, v in _casci(case, h, eri, tuples).items()})
        inc = _increments(eps, e_ref, orders)
    return orders, eps, inc, e_ref


def exact(case, seed):
    # the solves that would take too long are left out
    if case["kind"] != "sigma":
        cost = sum(_ndet(*s) * float(s[0]) ** 4 for s in _sizes(case))
        if cost > 6e10 or (case["recipe"] == "chain" and cost > 2e10):
            return None
    dev = _dev()
    h, eri = (torch.from_numpy(x).to(dev) for x in _integrals(case, seed))
    na, nb = _occ(case)
    ref, exp = _spaces(case)
    if case["kind"] == "sigma":
        n, a, b = _sizes(case)[0]
        _, g = _effective(h, eri, nb, a + b, ref)
        sh = _Shape(n, a, b)
        c = torch.from_numpy(_vector(sh.oa.shape[0], seed)).to(dev)[None]
        return {"sigma": (sh.h(g[None], c) + SPIN_SHIFT * sh.s2(c))[0]}
    if case["kind"] == "solve":
        tuples = _tuples(case, seed)
        res = _casci(case, h, eri, tuples)
        return {"eps": np.array([res[t][0] for t in tuples]), "status": None}
    if case["kind"] == "expand":
        orders, eps, inc, e_ref = _screened(case, h, eri)
        e_order = [math.fsum(inc[t] for t in o) for o in orders]
        flat = [t for o in orders for t in o]
        return _expansion(e_ref, e_order, math.fsum([e_ref] + e_order),
                          np.array([eps[t] for t in flat]), np.array([inc[t] for t in flat]), None)
    # grad: the expansion is linear in the tuple energies, each stationary in
    # its vector, so the derivative of sum_T c_T <x_T|H(h, eri)|x_T> is taken
    # with the vectors fixed
    sets = [t for k in range(case["order"] + 1) for t in itertools.combinations(exp, k)]
    res = _casci(case, h, eri, sets)
    coef = {t: 0 for t in sets}
    for t in sets:
        for k in range(len(t) + 1):
            for s in itertools.combinations(t, k):
                coef[s] += (-1) ** (len(t) - k)
    energy = math.fsum(coef[t] * res[t][0] for t in sets)
    gh, ge = torch.zeros_like(h), torch.zeros_like(eri)
    shapes = {}
    for t in sets:
        if coef[t] == 0:
            continue
        _, x, key = res[t]
        sh = shapes.setdefault(key, _Shape(*key))
        D = sh.D(x[None])[0].reshape(key[0] * (key[0] + 1) // 2, -1)
        gram = D @ D.T
        hh, ee = h.clone().requires_grad_(), eri.clone().requires_grad_()
        ecore, g = _effective(hh, ee, nb, key[1] + key[2], sorted(ref + list(t)))
        d = torch.autograd.grad(ecore + 0.5 * (g * gram).sum(), (hh, ee))
        gh += coef[t] * d[0]
        ge += coef[t] * d[1]
    return {"energy": np.float64(energy), "dh": 0.5 * (gh + gh.T), "deri": 0.5 * (ge + ge.T)}
