"""Every kernel of the grouped products on lists that the rules on sizes would give to another
one (GPU): the FP64 FMA tiles, the digit-product tiles of a CTA and of a warp, and the split-TF32
form, chosen through `Context.set_kernels`.  The launch counts say which kernel ran, so a rule
that moves cannot take a test off the kernel it is for."""
import numpy as np
import pytest

import synth
from oracle import blocks as ob
from oracle import dmrg, fock
from oracle import mps as om
from oracle import tda

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RTOL = 1e-12         # FP64 sigma, relative to max|y|
MIXED_RTOL = 1e-5    # split TF32, as in test_gpu_mixed.py
KERNELS = (1, 2, 3)  # FP64 FMA, digits by CTA tiles, by warp tiles


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_1646_gb300 import build
    build.build()
    import paper_1311_1646_gb300 as p
    p.load()
    return p


def _context(pkg, H, m, i, nsite, kernel=0, mixed=False, prec=0, scale=1.0):
    ctx = pkg.Context(0)
    ctx.set_kernels(kernel, mixed)
    ctx.op_build(H.k, H.h * scale, H.eri * scale)
    ctx.mps_load(H.k, H.n_alpha, H.n_beta, m.bonds, m.sites, i)
    for b in range(i):
        ctx.renormalize(b, +1, prec)
    for b in range(H.k - 1, i + nsite - 1, -1):
        ctx.renormalize(b, -1, prec)
    return ctx


def _sigma(ctx, i, nsite, x, nvec, prec=0):
    xd = torch.tensor(x, dtype=torch.float64, device="cuda:0")
    yd = torch.full_like(xd, float("nan"))
    ctx.sigma(i, nsite, xd, yd, nvec=nvec, precision=prec)
    torch.cuda.synchronize()
    return yd.cpu().numpy()


def _only(ctx, kernel):
    n = ctx.kernel_launches()
    return n[kernel - 1] > 0 and sum(n) == n[kernel - 1]


def _oracle(H, m, i, nsite):
    t, v = fock.spin_integrals(H.h, H.eri)
    env = ob.Environment(H, t, v)
    sites = [om.unpack_site(m.sites[j], m.bonds[j], m.bonds[j + 1]) for j in range(H.k)]
    for b in range(i):
        env.grow_left(b, sites[b])
    for b in range(H.k - 1, i + nsite - 1, -1):
        env.grow_right(b, sites[b])
    b = m.bonds

    def apply(x):
        if nsite == 1:
            w = om.unpack_site(x, b[i], b[i + 1])
            return om.pack_site(ob.sigma_onesite(env, i, w), b[i], b[i + 1])
        w = om.unpack_twosite(x, b[i], b[i + 2])
        return om.pack_twosite(ob.sigma_twosite(env, i, w), b[i], b[i + 2])
    return apply


# sectors of 1 to 66 states: row and column tiles of 1, of just below, at and above 16s, chunks of
# one and of many segments, split and whole segment lists; renormalization, one and two sites
@pytest.mark.parametrize("k,na,nb,M,i,nsite,nvec", [
    (6, 3, 3, 20, 0, 1, 2), (12, 1, 1, 3, 5, 1, 1), (8, 1, 1, 17, 3, 1, 2), (10, 2, 1, 60, 4, 1, 3), (9, 1, 2, 96, 4, 2, 1),
    (9, 4, 4, 60, 4, 2, 3), (10, 2, 2, 131, 4, 1, 5), (10, 2, 2, 190, 5, 2, 2)])
def test_sigma_of_every_kernel_matches_the_oracle(pkg, k, na, nb, M, i, nsite, nvec):
    H = synth.ab_initio(k, na, nb, 60 + M)
    m = synth.mixed_mps(k, na, nb, M, 61, center=i)
    ref = _oracle(H, m, i, nsite)
    n = x = r = None
    for kernel in KERNELS:
        ctx = _context(pkg, H, m, i, nsite, kernel)
        if x is None:
            n, _ = ctx.wfn_layout(i, nsite)
            x = synth.random_vector(nvec * n, 62)
            r = [ref(x[v * n:(v + 1) * n]) for v in range(nvec)]
        y = _sigma(ctx, i, nsite, x, nvec)
        for v in range(nvec):
            assert np.abs(y[v * n:(v + 1) * n] - r[v]).max() <= RTOL * np.abs(r[v]).max(), (kernel, v)
            # a vector's bits do not depend on the others in the call
            assert np.array_equal(_sigma(ctx, i, nsite, x[v * n:(v + 1) * n], 1), y[v * n:(v + 1) * n]), (kernel, v)
        assert _only(ctx, kernel), (kernel, ctx.kernel_launches())
        ctx.close()


@pytest.mark.parametrize("kernel", [2, 3])
def test_far_exponents_and_infinities_of_the_digit_kernels(pkg, kernel):
    """H scaled by 2^-500 leaves the integer path's exponents: plain FP64 from the staged
    operands, equal after rescaling to the rounding of either (1e-13).  An infinity or a NaN in
    one vector reaches its own result only."""
    k, na, nb, M, i = 10, 2, 2, 131, 4
    H = synth.ab_initio(k, na, nb, 7)
    m = synth.mixed_mps(k, na, nb, M, 8, center=i)
    a = _context(pkg, H, m, i, 1, kernel)
    n, _ = a.wfn_layout(i, 1)
    x = synth.random_vector(2 * n, 9)
    y = _sigma(a, i, 1, x, 2)
    b = _context(pkg, H, m, i, 1, kernel, scale=2.0 ** -500)
    z = _sigma(b, i, 1, x, 2) * 2.0 ** 500
    assert np.abs(z - y).max() <= 1e-13 * np.abs(y).max()
    for bad in (np.inf, np.nan):
        x2 = x.copy()
        x2[n // 2] = bad
        w = _sigma(a, i, 1, x2, 2)
        assert not np.all(np.isfinite(w[:n]))
        assert np.array_equal(w[n:], y[n:])
    assert _only(a, kernel) and _only(b, kernel)
    a.close()
    b.close()


@pytest.mark.parametrize("kernel", KERNELS)
def test_batches_of_every_kernel_match_single_calls(pkg, kernel):
    """Merged lists (uneven molecules, one and two sites) against each instance's own call on the
    FP64 FMA tiles; the second and third calls replay the captured graph."""
    for nsite in (1, 2):
        ctxs, xs, ys, refs, sites = [], [], [], [], []
        for j, (k, na, nb, M) in enumerate([(6, 3, 3, 20), (7, 2, 3, 33), (8, 2, 2, 48)]):
            H = synth.ab_initio(k, na, nb, 70 + j)
            i = k // 2 - 1
            m = synth.mixed_mps(k, na, nb, M, 71 + j, center=i)
            plain = _context(pkg, H, m, i, nsite, 1)
            n, _ = plain.wfn_layout(i, nsite)
            x = synth.random_vector(3 * n, 72 + j)
            refs.append(_sigma(plain, i, nsite, x, 3))
            plain.close()
            ctxs.append(_context(pkg, H, m, i, nsite, kernel))
            xs.append(torch.tensor(x, dtype=torch.float64, device="cuda:0"))
            ys.append(torch.full_like(xs[-1], float("nan")))
            sites.append(i)
        for _ in range(3):
            for y in ys:
                y.fill_(float("nan"))
            pkg.sigma_batched(ctxs, sites, nsite, xs, ys, nvec=3)
            torch.cuda.synchronize()
            for y, r in zip(ys, refs):
                assert np.abs(y.cpu().numpy() - r).max() <= RTOL * np.abs(r).max()
        assert _only(ctxs[0], kernel), ctxs[0].kernel_launches()
        for c in ctxs:
            c.close()


def _stationary(k, na, nb, M):
    H = synth.ab_initio(k, na, nb, 7)
    t, v = fock.spin_integrals(H.h, H.eri)
    _, sites, _ = dmrg.ground_state(H, t, v, [M], synth.random_mps(k, na, nb, M, 3))
    _, sites, _ = dmrg.onesite_sweeps(H, t, v, sites, n_sweeps=30, dav_tol=1e-13)
    return H, om.mixed_canonical(sites)


@pytest.fixture(scope="module")
def reference_k5():
    k, na, nb, M, n = 5, 3, 2, 10, 3
    H, ref = _stationary(k, na, nb, M)
    L0, R0, C0, Lam, _ = ref
    w, E0, _ = tda.tangent_rr(H, L0, R0, C0, Lam, n)
    return H, ref, w, E0, n


def _tda(pkg, H, ref, n, kernel=0, mixed=False, **kw):
    L0, R0, C0, Lam, _ = ref
    k = H.k
    tables = [[(q[0], q[1], len(Lam[b][q])) for q in sorted(Lam[b])] for b in range(k + 1)]
    pack = [[om.pack_site(T[i], tables[i], tables[i + 1]) for i in range(k)] for T in (L0, R0, C0)]
    lam = [np.concatenate([Lam[b][q] for q in sorted(Lam[b])]) for b in range(k + 1)]
    ctx = pkg.Context(0)
    ctx.set_kernels(kernel, mixed)
    ctx.op_build(k, H.h, H.eri, e_core=H.e_core)
    ctx.mps_load(k, H.n_alpha, H.n_beta, tables, pack[0], 0, sites_right=pack[1])
    ctx.tda_load(pack[2], lam)
    out = ctx.sweep_tda(n, **kw)
    counts = ctx.kernel_launches()
    ctx.close()
    return out, counts


@pytest.mark.parametrize("kernel", KERNELS)
def test_tda_replays_of_every_kernel_reach_the_roots(pkg, reference_k5, kernel):
    """The kept plans replayed over the trial vectors (the kernels' instance forms)."""
    H, ref, w, E0, n = reference_k5
    (omega, resid, e0), counts = _tda(pkg, H, ref, n, kernel, max_iter=150, eps=1e-10, keep=6, max_space=18)
    assert abs(e0 - E0) < 1e-10 and np.all(resid < 1e-10)
    assert np.abs(omega + e0 - w).max() < 1e-8
    assert counts[kernel - 1] > 0 and sum(counts) == counts[kernel - 1], counts


def test_tda_on_split_tf32_reaches_the_roots(pkg, reference_k5):
    H, ref, w, E0, n = reference_k5
    (omega, resid, e0), counts = _tda(pkg, H, ref, n, 0, True, max_iter=150, eps=1e-10, keep=6, max_space=18, precision=1)
    assert np.all(resid < 1e-10)
    assert np.abs(omega + e0 - w).max() < 1e-6
    assert counts[3] > 0, counts


# two-site and one-site split-TF32 lists of narrow blocks, several vectors
@pytest.mark.parametrize("cfg,i,nsite,nvec", [(0, 0, 1, 2), (0, 2, 2, 2), (0, 5, 1, 1), (1, 3, 2, 3), (2, 5, 2, 6)])
def test_split_tf32_sigma_matches_fp64(pkg, cfg, i, nsite, nvec):
    H, M = (synth.ab_initio(6, 3, 3, 21), 20) if cfg == 0 else (synth.config(cfg)["ham"], synth.config(cfg)["M"])
    m = synth.mixed_mps(H.k, H.n_alpha, H.n_beta, M, 300 + cfg, center=i)
    ctx = _context(pkg, H, m, i, nsite, 0, True)
    n, _ = ctx.wfn_layout(i, nsite)
    x = synth.random_vector(nvec * n, 7)
    a, b = _sigma(ctx, i, nsite, x, nvec), _sigma(ctx, i, nsite, x, nvec, 1)
    assert ctx.kernel_launches()[3] == 2 and not np.array_equal(a, b)
    assert np.abs(a - b).max() <= MIXED_RTOL * np.abs(a).max()
    ctx.close()


@pytest.mark.parametrize("cfg,i,nsite", [(1, 3, 2), (2, 5, 2)])
def test_split_tf32_renormalization(pkg, cfg, i, nsite):
    c = synth.config(cfg)
    H = c["ham"]
    m = synth.mixed_mps(H.k, H.n_alpha, H.n_beta, c["M"], 400 + cfg, center=i)
    out = []
    for prec in (0, 1):
        ctx = _context(pkg, H, m, i, nsite, 0, True, prec)
        assert (ctx.kernel_launches()[3] > 0) == (prec == 1)
        n, _ = ctx.wfn_layout(i, nsite)
        out.append(_sigma(ctx, i, nsite, synth.random_vector(n, 8), 1))
        ctx.close()
    assert 0.0 < np.abs(out[0] - out[1]).max() <= 5e-5 * np.abs(out[0]).max()


def test_split_tf32_batch_matches_fp64(pkg):
    ctxs, xs, ys, refs, sites = [], [], [], [], []
    for j, (k, na, nb, M) in enumerate([(6, 3, 3, 20), (7, 2, 3, 33), (8, 2, 2, 48)]):
        H = synth.ab_initio(k, na, nb, 70 + j)
        i = k // 2 - 1
        m = synth.mixed_mps(k, na, nb, M, 71 + j, center=i)
        c = _context(pkg, H, m, i, 1, 0, True)
        n, _ = c.wfn_layout(i, 1)
        x = synth.random_vector(2 * n, 72 + j)
        refs.append(_sigma(c, i, 1, x, 2))
        ctxs.append(c)
        xs.append(torch.tensor(x, dtype=torch.float64, device="cuda:0"))
        ys.append(torch.full_like(xs[-1], float("nan")))
        sites.append(i)
    for _ in range(3):
        pkg.sigma_batched(ctxs, sites, 1, xs, ys, nvec=2, precision=1)
        torch.cuda.synchronize()
        for y, r in zip(ys, refs):
            e = np.abs(y.cpu().numpy() - r).max()
            assert 0.0 < e <= MIXED_RTOL * np.abs(r).max()
    assert ctxs[0].kernel_launches()[3] == 6
    for c in ctxs:
        c.close()


def test_split_tf32_runs_again_after_an_expired_wait(pkg):
    """After a wait that ran out (test hook, 20 ms limit), the next calls run on the same kernels."""
    c = synth.config(1)
    H, i = c["ham"], 3
    m = synth.mixed_mps(H.k, H.n_alpha, H.n_beta, c["M"], 31, center=i)
    ctx = _context(pkg, H, m, i, 1, 0, True)
    n, _ = ctx.wfn_layout(i, 1)
    x = synth.random_vector(2 * n, 41)
    ref = _sigma(ctx, i, 1, x, 2)
    first = _sigma(ctx, i, 1, x, 2, 1)
    ctx.set_wait_limit(0.02, stall_next=True)
    with pytest.raises(pkg.LrtError, match=r"\(-5\)"):
        _sigma(ctx, i, 1, x, 2, 1)
    before = ctx.kernel_launches()[3]
    again = _sigma(ctx, i, 1, x, 2, 1)
    assert ctx.kernel_launches()[3] == before + 2
    for y in (first, again):
        assert 0.0 < np.abs(y - ref).max() <= MIXED_RTOL * np.abs(ref).max()
    ctx.set_wait_limit(0.0)
    ctx.close()
