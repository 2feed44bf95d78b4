"""Timed cases of the DMRG effective-Hamiltonian library: what a program does with it.

Each case is one call, or the few calls of one sweep position, through the package's public
entry points (`Context`, `sigma_batched`): the effective-Hamiltonian sigma vector on one- and
two-site tensors, block renormalization with the diagonal and the first sigma at the next
position, independent small molecules in one batched call, a ground-state run and a few
tangent-space (TDA) sweeps.  Every input is drawn from the seed: integrals, isometries and
trial vectors.  Trial vectors carry a decaying weight per right state of a sector, as
wavefunctions in a Schmidt basis do.
"""
import math

import numpy as np

QN = ((0, 0), (1, 0), (0, 1), (1, 1))   # (N_alpha, N_beta) of the site states |0>, |a>, |b>, |ab>


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def _c(name, kind, ham, k, na, nb, M, site, nsite=1, nvec=1, prec="fp64", direction=1, count=1):
    c = dict(kind=kind, ham=ham, k=k, na=na, nb=nb, M=M, site=site, nsite=nsite, nvec=nvec, prec=prec,
             direction=direction, count=count)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call in earnest: one Davidson product of the 8-orbital active space
        _c("sigma1_k8_M64", "sigma", "ab", 8, 4, 4, 64, 3),
        # the ground-state Davidson's product at the middle of the 12-site polyene
        _c("sigma2_ppp_k12_M256", "sigma", "ppp", 12, 6, 6, 256, 5, nsite=2),
        # block Davidson of 6 roots on the water-shaped workload (the benchmark's call)
        _c("sigma1_water_k24_M500_6vec", "sigma", "water", 24, 5, 5, 500, 11, nvec=6),
        # the same workload near an end of the chain, one vector: few, uneven sectors
        _c("sigma1_water_k24_M300_edge", "sigma", "water", 24, 5, 5, 300, 4),
        # the mixed (split-TF32) form of the benchmark's call
        _c("sigma1_water_k24_M500_6vec_mixed", "sigma", "water", 24, 5, 5, 500, 11, nvec=6, prec="mixed"),
        # two-site, odd orbital and electron counts, odd vector count, mixed
        _c("sigma2_k13_M200_3vec_mixed", "sigma", "ab", 13, 7, 6, 200, 5, nsite=2, nvec=3, prec="mixed"),
        # one position of a two-site ground-state sweep to the right: renormalize, diagonal, product
        _c("step2_right_k12_M128", "step", "ab", 12, 6, 6, 128, 5, nsite=2, direction=1),
        # one position of a one-site sweep to the left, larger blocks, 4 vectors
        _c("step1_left_k16_M384_4vec", "step", "ab", 16, 8, 8, 384, 8, nvec=4, direction=-1),
        # eight independent small molecules of uneven sizes in one call
        _c("batch8_k8to12_4vec", "batch", "ab", 8, 4, 4, 96, 0, nvec=4, count=8),
        # the two first ground-state sweeps of the 8-orbital active space, as one call
        _c("sweep_gs_k8_M64", "gs", "ab", 8, 4, 4, 64, 0),
        # two tangent-space sweeps for 6 roots on the polyene, after the start sweep
        _c("sweep_tda_ppp_k12_M128_6roots", "tda", "ppp", 12, 6, 6, 128, 0, nvec=6),
    ]


def draw(rng):
    """One more case: sizes over the ranges of the listed ones, uneven fillings and odd counts
    among them; at most the work of the 24-orbital call."""
    kind = rng.choice(["sigma"] * 6 + ["step"] * 3 + ["batch"])
    k = rng.randint(6, 18)
    n = k + rng.choice([-3, -2, -1, 0, 0, 1, 2])
    na = max(1, min(k, n // 2 + rng.choice([0, 0, 1])))
    nb = max(1, min(k, n - na))
    M = int(round(math.exp(rng.uniform(math.log(12), math.log(420 if k <= 14 else 260)))))
    nsite = rng.choice([1, 1, 2])
    nvec = rng.choice([1, 1, 2, 3, 4, 5, 6, 8])
    prec = rng.choice(["fp64", "fp64", "mixed"])
    if kind == "batch":
        return _c(None, kind, "ab", rng.randint(6, 9), 3, rng.randint(2, 3), rng.randint(12, 120), 0, nsite, nvec, prec,
                  count=rng.randint(3, 10))
    if kind == "step":
        d = rng.choice([1, -1])
        lo, hi = (0, k - nsite - 1) if d == 1 else (nsite, k - 1)
        return _c(None, kind, "ab", k, na, nb, M, (rng.randint(lo, hi) + rng.randint(lo, hi)) // 2, nsite, nvec, "fp64", d)
    site = (rng.randint(0, k - nsite) + rng.randint(0, k - nsite)) // 2   # the middle more often than the ends
    return _c(None, kind, rng.choice(["ab", "ab", "ab", "water"]), k, na, nb, M, site, nsite, nvec, prec)


# ---------------------------------------------------------------------------------------
# inputs (plain numpy, from the seed alone)
# ---------------------------------------------------------------------------------------
def _count(n, a, b):
    return 0 if a < 0 or b < 0 or a > n or b > n else math.comb(n, a) * math.comb(n, b)


def _bonds(k, na, nb, M):
    """Bond tables [(N_alpha left, N_beta left, states)]: the exact sector sizes, shared out in
    proportion where their sum exceeds M, every sector reachable from its neighbours."""
    tabs = []
    for b in range(k + 1):
        exact = {}
        for a in range(min(b, na) + 1):
            for c in range(min(b, nb) + 1):
                d = min(_count(b, a, c), _count(k - b, na - a, nb - c))
                if d:
                    exact[(a, c)] = d
        tot = sum(exact.values())
        if tot > M:
            exact = {q: max(1, min(e, int(M * e / tot))) for q, e in exact.items()}
        tabs.append(exact)
    for _ in range(2):
        for b in range(1, k + 1):
            for q in tabs[b]:
                tabs[b][q] = min(tabs[b][q], sum(tabs[b - 1].get((q[0] - s[0], q[1] - s[1]), 0) for s in QN))
        for b in range(k - 1, -1, -1):
            for q in tabs[b]:
                tabs[b][q] = min(tabs[b][q], sum(tabs[b + 1].get((q[0] + s[0], q[1] + s[1]), 0) for s in QN))
        tabs = [{q: d for q, d in t.items() if d > 0} for t in tabs]
    return [[(q[0], q[1], d) for q, d in sorted(t.items())] for t in tabs]


def _layout(left, right):
    """[(q_l, n, q_r, D_l, D_r, offset)] of a site tensor: per right sector, sub-blocks n = 0..3."""
    ld = {(a, b): d for a, b, d in left}
    out, off = [], 0
    for a, b, dr in right:
        for n, s in enumerate(QN):
            q = (a - s[0], b - s[1])
            if q in ld:
                out.append((q, n, (a, b), ld[q], dr, off))
                off += ld[q] * dr
    return out, off


def _ortho(G):
    Q, R = np.linalg.qr(G)
    s = np.sign(np.diag(R))
    return Q * np.where(s == 0, 1.0, s)


def _site(rng, left, right, form):
    """A random site tensor: left-orthonormal columns of every fused block, or right-orthonormal
    rows of every right-fused one."""
    lay, size = _layout(left, right)
    a = rng.standard_normal(size)
    groups = {}
    for e in lay:
        groups.setdefault(e[2] if form == "left" else e[0], []).append(e)
    for es in groups.values():
        blocks = [a[e[5]:e[5] + e[3] * e[4]].reshape(e[3], e[4]) for e in es]
        G = np.vstack(blocks) if form == "left" else np.hstack(blocks).T
        Q = _ortho(G)
        r = 0
        for e in es:
            m = e[3] if form == "left" else e[4]
            part = Q[r:r + m] if form == "left" else Q[r:r + m].T
            a[e[5]:e[5] + e[3] * e[4]] = part.ravel()
            r += m
    return a


def _hamiltonian(rng, ham, k):
    """(h, eri, e_core).  "ab": random one-body part on a rising diagonal, two-body part from k
    factors; "water": the factors decay as exp(-|i-j| / 6); "ppp": trans-polyene with the Ohno
    interaction (bonds 1.35 / 1.46 A, t = -2.4 / -2.2 eV, U = 11.13 eV), no random part."""
    if ham == "ppp":
        pos = np.zeros((k, 2))
        h = np.zeros((k, k))
        for b in range(k - 1):
            ang = math.radians(30.0 if b % 2 == 0 else -30.0)
            pos[b + 1] = pos[b] + (1.35 if b % 2 == 0 else 1.46) * np.array([math.cos(ang), math.sin(ang)])
            h[b, b + 1] = h[b + 1, b] = -2.4 if b % 2 == 0 else -2.2
        eri = np.zeros((k,) * 4)
        core = 0.0
        for i in range(k):
            for j in range(k):
                V = 11.13 / math.sqrt(1.0 + (11.13 * float(np.linalg.norm(pos[i] - pos[j])) / 14.397) ** 2)
                eri[i, i, j, j] = V
                if i != j:
                    h[i, i] -= V
                    core += 0.5 * V
        ev = 1.0 / 27.211386
        return h * ev, eri * ev, core * ev
    h = 0.5 * rng.standard_normal((k, k))
    h = np.triu(h) + np.triu(h, 1).T + np.diag(np.linspace(-2.0, 0.0, k))
    B = 0.3 * rng.standard_normal((k, k, k))
    B = np.triu(B) + np.transpose(np.triu(B, 1), (0, 2, 1))
    if ham == "water":
        i = np.arange(k)
        B = B * np.exp(-np.abs(i[:, None] - i[None, :]) / 6.0)
    F = B.reshape(k, k * k)
    return h, (F.T @ F).reshape(k, k, k, k), 0.0


def _wave(rng, bonds, site, nsite, nvec):
    """Trial vectors, normalized, right states of a sector weighted from 1 down to 1e-4."""
    out = []
    for _ in range(nvec):
        parts = []
        if nsite == 1:
            lay, _ = _layout(bonds[site], bonds[site + 1])
            for (_, _, _, dl, dr, _) in lay:
                parts.append(rng.standard_normal((dl, dr)) * 10.0 ** (-4.0 * np.arange(dr) / max(dr, 2)))
        else:
            for (_, ls, rs) in _twosite(bonds[site], bonds[site + 2]):
                g = rng.standard_normal((sum(x[2] for x in ls), sum(x[2] for x in rs)))
                w = np.concatenate([10.0 ** (-4.0 * np.arange(x[2]) / max(x[2], 2)) for x in rs])
                parts.append(g * w)
        v = np.concatenate([p.ravel() for p in parts])
        out.append(v / np.linalg.norm(v))
    return np.concatenate(out)


def _twosite(left, right):
    """[(q_m, [(n1, q_l, D_l)], [(n2, q_r, D_r)])] of a two-site wavefunction, in storage order."""
    ld = {(a, b): d for a, b, d in left}
    rd = {(a, b): d for a, b, d in right}
    out = []
    for m in sorted({(q[0] + s[0], q[1] + s[1]) for q in ld for s in QN}):
        ls = [(n, (m[0] - s[0], m[1] - s[1])) for n, s in enumerate(QN)]
        rs = [(n, (m[0] + s[0], m[1] + s[1])) for n, s in enumerate(QN)]
        ls = [(n, q, ld[q]) for n, q in ls if q in ld]
        rs = [(n, q, rd[q]) for n, q in rs if q in rd]
        if ls and rs:
            out.append((m, ls, rs))
    return out


def _instance(case, j=0):
    """The shape of instance j of a batch (the case itself otherwise): 8 to 12 orbitals, fillings
    and bond dimensions varied, the middle site."""
    if case["kind"] != "batch":
        return case
    k = case["k"] + (3 * j) % 5
    na, nb = case["na"] + (j % 3), case["nb"] + (j % 2)
    return dict(case, k=k, na=min(na, k), nb=min(nb, k), M=case["M"] + 13 * ((5 * j) % 7), site=k // 2 - 1)


def _position(case):
    """(site, nsite) of the wavefunction: for a step, the position the sweep moves to."""
    if case["kind"] != "step":
        return case["site"], case["nsite"]
    return (case["site"] + 1 if case["direction"] == 1 else case["site"] - case["nsite"]), case["nsite"]


def _inputs(case, seed, j=0):
    c = _instance(case, j)
    rng = np.random.default_rng([int(seed), j, 1311])
    k, na, nb = c["k"], c["na"], c["nb"]
    h, eri, core = _hamiltonian(rng, c["ham"], k)
    bonds = _bonds(k, na, nb, c["M"])
    site, nsite = _position(c)
    if c["kind"] in ("gs", "tda"):
        start = bonds if c["kind"] == "tda" else _bonds(k, na, nb, 16)
        return c, h, eri, core, start, [_site(rng, start[i], start[i + 1], "right") for i in range(k)], None, 0, 1
    sites = [_site(rng, bonds[i], bonds[i + 1], "left" if i < site else "right") for i in range(k)]
    x = _wave(rng, bonds, site, nsite, c["nvec"])
    return c, h, eri, core, bonds, sites, x, site, nsite


# ---------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------------------
def _context(case, seed, j=0):
    import torch

    import paper_1311_1646_gb300 as pkg
    c, h, eri, core, bonds, sites, x, site, nsite = _inputs(case, seed, j)
    k = c["k"]
    ctx = pkg.Context(0)
    ctx.op_build(k, h, eri, e_core=core)
    ctx.mps_load(k, c["na"], c["nb"], bonds, sites, site)
    s = dict(case=c, ctx=ctx, pkg=pkg, torch=torch, site=site, nsite=nsite, bonds=bonds, sites=sites)
    if c["kind"] == "tda":
        ctx.tda_prepare()
    if x is None:
        return s
    for b in range(site):
        ctx.renormalize(b, +1)
    for b in range(k - 1, site + nsite - 1, -1):
        ctx.renormalize(b, -1)
    s["x"] = torch.from_numpy(x).cuda()
    s["y"] = torch.empty_like(s["x"])
    s["d"] = torch.empty(s["x"].numel() // c["nvec"], dtype=torch.float64, device="cuda")
    s["prec"] = pkg.LRT_MIXED if c["prec"] == "mixed" else pkg.LRT_FP64
    return s


def prepare(case, seed):
    if case["kind"] == "batch":
        return [_context(case, seed, j) for j in range(case["count"])]
    return _context(case, seed)


def _result(s, y):
    # the mixed form carries about seven digits: its caller keeps the product in 32 bits
    return y.float() if s["prec"] == s["pkg"].LRT_MIXED else y


def run(state):
    if isinstance(state, list):
        s = state[0]
        s["pkg"].sigma_batched([t["ctx"] for t in state], [t["site"] for t in state], s["nsite"], [t["x"] for t in state],
                               [t["y"] for t in state], nvec=s["case"]["nvec"], precision=s["prec"])
        return [_result(t, t["y"]) for t in state]
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "gs":
        ctx.mps_load(c["k"], c["na"], c["nb"], state["bonds"], state["sites"], 0)
        return ctx.sweep_gs([16, c["M"]], max_sweeps=2, sweeps_per_M=1, e_tol=1e-10, dav_tol=1e-8)
    if c["kind"] == "tda":
        omega, resid, e0 = ctx.sweep_tda(c["nvec"], max_iter=2, eps=1e-30, allow_noconv=True, max_space=32,
                                         keep=2 * c["nvec"], correction=1, start_shift=0.1)
        return {"omega": omega, "resid": resid, "e0": e0}
    if c["kind"] == "step":
        ctx.renormalize(c["site"], c["direction"])
        ctx.heff_diag(state["site"], state["nsite"], state["d"])
        ctx.sigma(state["site"], state["nsite"], state["x"], state["y"], nvec=c["nvec"])
        return {"diag": state["d"], "sigma": state["y"]}
    ctx.sigma(state["site"], state["nsite"], state["x"], state["y"], nvec=c["nvec"], precision=state["prec"])
    return _result(state, state["y"])


# ---------------------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------------------
def _operators(nl, k, normal):
    """{(dN_alpha, dN_beta): count} of the renormalized operators of a block of nl orbitals: the
    identity and H, creators, three-index operators, and the pair operators of its own orbitals
    (normal) or of the others (complementary)."""
    out = {}

    def add(a, b, n):
        if n:
            out[(a, b)] = out.get((a, b), 0) + n
    m = nl if normal else k - nl
    add(0, 0, 2)
    for s in ((1, 0), (0, 1)):
        add(s[0], s[1], nl)
        add(-s[0], -s[1], k - nl)
    sg = 1 if normal else -1
    add(2 * sg, 0, m * (m - 1) // 2)
    add(0, 2 * sg, m * (m - 1) // 2)
    add(sg, sg, m * m)
    add(0, 0, m * (m + 1))
    add(sg, -sg, m * (m + 1) // 2)
    add(-sg, sg, m * (m - 1) // 2)
    return out


def _set_size(tab, ops, sign):
    dim = {(a, b): d for a, b, d in tab}
    return sum(n * d * dim.get((q[0] + sign * o[0], q[1] + sign * o[1]), 0) for o, n in ops.items() for q, d in dim.items())


def _sigma_work(c, site, nsite):
    """Operator blocks of both sides read once, x read and y written; products: every operator
    (and its adjoint) of the side that holds the pair operators applied to x, and its partner
    applied to the result."""
    k, bonds = c["k"], _bonds(c["k"], c["na"], c["nb"], c["M"])
    bl, br = site, site + nsite
    lops = _operators(bl, k, 2 * bl <= k)
    rops = _operators(k - br, k, 2 * br > k)
    ld = {(a, b): d for a, b, d in bonds[bl]}
    rd = {(a, b): d for a, b, d in bonds[br]}
    steps = [((s[0] + t[0], s[1] + t[1])) for s in QN for t in (QN if nsite == 2 else QN[:1])]
    n = sum(d * rd.get((q[0] + s[0], q[1] + s[1]), 0) for q, d in ld.items() for s in steps)
    m = min(site + 1, k - site - 1)
    # the polyene's two-body part couples densities only: one operator per spin orbital and its hops
    pairs = {(0, 0): 2 + 2 * m, (1, 0): 2, (0, 1): 2} if c["ham"] == "ppp" else _operators(m, k, True)
    flops = 0.0
    for o, cnt in pairs.items():
        for sg in (1, -1):
            for q, d in ld.items():
                for s in steps:
                    dr = rd.get((q[0] + s[0], q[1] + s[1]), 0)
                    dl2 = ld.get((q[0] + sg * o[0], q[1] + sg * o[1]), 0)
                    dr2 = rd.get((q[0] + s[0] + sg * o[0], q[1] + s[1] + sg * o[1]), 0)
                    flops += 2.0 * cnt * dl2 * dr * (d + dr2)
    nb = 8.0 * (_set_size(bonds[bl], lops, 1) + _set_size(bonds[br], rops, -1) + 2 * n * c["nvec"])
    return {"bytes": nb, "flops": flops * c["nvec"]}


def work(case):
    tot = {"bytes": 0.0, "flops": 0.0}
    for j in range(case["count"]):
        c = _instance(case, j)
        k, bonds = c["k"], _bonds(c["k"], c["na"], c["nb"], c["M"])
        site, nsite = _position(c)
        if c["kind"] in ("gs", "tda"):
            # one product per position and sweep direction (TDA: per root), the least of any sweep
            sweeps = 2 if c["kind"] == "gs" else 3
            for i in range(k - 1):
                w = _sigma_work(c, i, 2 if c["kind"] == "gs" else 1)
                for t in tot:
                    tot[t] += 2 * sweeps * w[t]
            continue
        w = _sigma_work(c, site, nsite)
        if c["kind"] == "step":
            # the new block written, the old one read, and the two-sided transformation by the site
            s, d = c["site"], c["direction"]
            new, old = (s + 1, s) if d == 1 else (s, s + 1)
            ops = _operators(new if d == 1 else k - new, k, (2 * new <= k) == (d == 1))
            M2, M1 = (sum(x[2] for x in bonds[b]) for b in (new, old))
            size = _set_size(bonds[new], ops, d)
            w["bytes"] += 8.0 * (size + _set_size(bonds[old], _operators(old if d == 1 else k - old, k, (2 * old <= k) == (d == 1)), d))
            w["flops"] += 4.0 * size * (M1 + M2) / max(1, len(bonds[old]))
        for t in tot:
            tot[t] += w[t]
    return tot


# ---------------------------------------------------------------------------------------
# the same products in 64 bits, in the space of determinants
# ---------------------------------------------------------------------------------------
def _strings(n, m):
    """The n-orbital strings of m electrons, ascending, and the place of each."""
    s = [b for b in range(1 << n) if bin(b).count("1") == m]
    return s, {b: i for i, b in enumerate(s)}


def _basis(bonds, sites, upto, k, left):
    """States of the block left (or right) of bond `upto` over its site-ordered determinants:
    {sector: (D x determinants, [(alpha bits, beta bits)])}."""
    if left:
        cur = {(0, 0): (np.ones((1, 1)), [(0, 0)])}
        rng = range(upto)
    else:
        a, b, _ = bonds[k][0]
        cur = {(a, b): (np.ones((1, 1)), [(0, 0)])}
        rng = range(k - 1, upto - 1, -1)
    for i in rng:
        lay, _ = _layout(bonds[i], bonds[i + 1])
        new = {}
        for ql, n, qr, dl, dr, off in lay:
            A = sites[i][off:off + dl * dr].reshape(dl, dr)
            src, dst, T = (ql, qr, A.T) if left else (qr, ql, A)
            C, dets = cur[src]
            add = [(p | (QN[n][0] << i), q | (QN[n][1] << i)) for p, q in dets]
            P, D = new.setdefault(dst, ([], []))
            P.append(T @ C)
            D.extend(add)
        cur = {q: (np.hstack(P), D) for q, (P, D) in new.items()}
    return cur


def _fci(h, eri, core, k, na, nb):
    """H as a function on the (alpha string, beta string) coefficient matrix, and the strings."""
    def excitations(strings, place):
        out = []
        for p in range(k):
            for q in range(k):
                src, dst, sg = [], [], []
                for s, b in enumerate(strings):
                    if not (b >> q) & 1:
                        continue
                    t = b & ~(1 << q)
                    if (t >> p) & 1:
                        continue
                    par = bin(b & ((1 << q) - 1)).count("1") + bin(t & ((1 << p) - 1)).count("1")
                    src.append(s)
                    dst.append(place[t | (1 << p)])
                    sg.append(-1.0 if par & 1 else 1.0)
                out.append((np.array(src, int), np.array(dst, int), np.array(sg)))
        return out
    sa, pa = _strings(k, na)
    sb, pb = _strings(k, nb)
    Ea, Eb = excitations(sa, pa), excitations(sb, pb)
    g = h - 0.5 * np.einsum("ijjl->il", eri)
    V = eri.reshape(k * k, k * k)

    def apply(C):
        D = np.zeros((k * k,) + C.shape)
        for t in range(k * k):
            s, d, sg = Ea[t]
            D[t][d] += sg[:, None] * C[s]
            s, d, sg = Eb[t]
            D[t][:, d] += sg[None, :] * C[:, s]
        G = (0.5 * V @ D.reshape(k * k, -1)).reshape(D.shape) + 0.0
        G += g.reshape(k * k)[:, None, None] * C
        out = core * C
        for t in range(k * k):
            s, d, sg = Ea[t]
            out[d] += sg[:, None] * G[t][s]
            s, d, sg = Eb[t]
            out[:, d] += sg[None, :] * G[t][:, s]
        return out
    return apply, pa, pb


def _sign(a, b):
    """Site order (0a 0b 1a 1b ...) to all alpha before all beta: one factor -1 for every beta
    electron left of an alpha one."""
    s = 0
    while a:
        low = a & -a
        s += bin(b & (low - 1)).count("1")
        a ^= low
    return -1.0 if s & 1 else 1.0


def _exact_sigma(c, h, eri, core, bonds, sites, x, site, nsite):
    k = c["k"]
    L = _basis(bonds, sites, site, k, True)
    R = _basis(bonds, sites, site + nsite, k, False)
    apply, pa, pb = _fci(h, eri, core, k, c["na"], c["nb"])
    # every piece of the wavefunction: (offset, row stride, q_l, q_r, bits of its sites)
    pieces = []
    if nsite == 1:
        lay, n = _layout(bonds[site], bonds[site + 1])
        for ql, n1, qr, dl, dr, off in lay:
            pieces.append((off, dr, ql, qr, dl, dr, QN[n1][0] << site, QN[n1][1] << site))
    else:
        n = 0
        for _, ls, rs in _twosite(bonds[site], bonds[site + 2]):
            cols, r0 = sum(t[2] for t in rs), 0
            for n1, ql, dl in ls:
                c0 = 0
                for n2, qr, dr in rs:
                    pieces.append((n + r0 * cols + c0, cols, ql, qr, dl, dr, (QN[n1][0] << site) | (QN[n2][0] << (site + 1)),
                                   (QN[n1][1] << site) | (QN[n2][1] << (site + 1))))
                    c0 += dr
                r0 += dl
            n += r0 * cols
    maps = []
    for off, ld, ql, qr, dl, dr, ba, bb in pieces:
        dets = [(p | ba | r, q | bb | s) for p, q in L[ql][1] for r, s in R[qr][1]]
        maps.append((np.array([pa[a] for a, _ in dets]), np.array([pb[b] for _, b in dets]), np.array([_sign(a, b) for a, b in dets])))
    out = []
    for v in range(c["nvec"]):
        xv = x[v * n:(v + 1) * n]
        C = np.zeros((len(pa), len(pb)))
        for (off, ld, ql, qr, dl, dr, _, _), (ia, ib, sg) in zip(pieces, maps):
            X = np.lib.stride_tricks.as_strided(xv[off:], (dl, dr), (8 * ld, 8))
            C[ia, ib] += sg * (L[ql][0].T @ X @ R[qr][0]).ravel()
        S = apply(C)
        y = np.zeros(n)
        for (off, ld, ql, qr, dl, dr, _, _), (ia, ib, sg) in zip(pieces, maps):
            W = (sg * S[ia, ib]).reshape(L[ql][0].shape[1], -1)
            np.lib.stride_tricks.as_strided(y[off:], (dl, dr), (8 * ld, 8))[:] = L[ql][0] @ W @ R[qr][0].T
        out.append(y)
    return np.concatenate(out)


def exact(case, seed):
    """The sigma vector by determinants; None for iterated results and where the determinants
    are too many (over a million per vector, or more than 3 million in all)."""
    if case["kind"] in ("gs", "tda"):
        return None
    res = []
    for j in range(case["count"]):
        c = _instance(case, j)
        nd = math.comb(c["k"], c["na"]) * math.comb(c["k"], c["nb"])
        if nd > 1.0e6 or nd * c["nvec"] > 3.0e6:
            res.append(None)
            continue
        c, h, eri, core, bonds, sites, x, site, nsite = _inputs(case, seed, j)
        res.append(_exact_sigma(c, h, eri, core, bonds, sites, x, site, nsite))
    if all(r is None for r in res):
        return None
    if case["kind"] == "batch":
        return res
    return {"diag": None, "sigma": res[0]} if case["kind"] == "step" else res[0]
