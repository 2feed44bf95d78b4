"""heff_diag prepares the single-vector plan of its position (GPU): the product that follows needs
no planning and can be captured; plans of other vector counts share its lists."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_1646_gb300 import build
    build.build()
    import paper_1311_1646_gb300 as p
    p.load()
    return p


def _context(pkg, H, M, i, nsite, seed, stream=None, kernel=0):
    m = synth.mixed_mps(H.k, H.n_alpha, H.n_beta, M, seed, center=i)
    ctx = pkg.Context(0, stream=stream)
    ctx.set_kernels(kernel)
    ctx.op_build(H.k, H.h, H.eri)
    ctx.mps_load(H.k, H.n_alpha, H.n_beta, m.bonds, m.sites, i)
    for b in range(i):
        ctx.renormalize(b, +1)
    for b in range(H.k - 1, i + nsite - 1, -1):
        ctx.renormalize(b, -1)
    return ctx


@pytest.mark.parametrize("noalloc", [True, False])
@pytest.mark.parametrize("first_nvec", [0, 3])
def test_first_product_after_heff_diag_is_captured(pkg, first_nvec, noalloc):
    cfg = synth.config(1)
    H, i = cfg["ham"], 3
    st = torch.cuda.Stream()
    ctx = _context(pkg, H, cfg["M"], i, 1, 77, st.cuda_stream)
    n, _ = ctx.wfn_layout(i, 1)
    with torch.cuda.stream(st):
        x = torch.tensor(synth.random_vector(3 * n, 5), dtype=torch.float64, device="cuda:0")
        y, d = torch.empty_like(x), torch.empty(n, dtype=torch.float64, device="cuda:0")
        out = torch.empty(n, dtype=torch.float64, device="cuda:0")
        if noalloc:      # the static array's address is resolved by a first call, at any position
            other = _context(pkg, H, 20, i, 1, 78, st.cuda_stream)
            k, _ = other.wfn_layout(i, 1)
            other.sigma(i, 1, x[:k], y[:k])
            other.sigma_noalloc(i, 1, x[:k], y[:k])
        if first_nvec:
            ctx.sigma(i, 1, x, y, nvec=3)
        ctx.heff_diag(i, 1, d)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):     # an allocation, copy or wait in the call would fail here
            (ctx.sigma_noalloc if noalloc else ctx.sigma)(i, 1, x[:n], out)
        out.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        ctx.sigma(i, 1, x[:n], out)
        torch.cuda.synchronize()
    assert np.array_equal(got, out.cpu().numpy())
    if noalloc:
        other.close()
    ctx.close()


@pytest.mark.parametrize("kernel", [0, 1, 2, 3])
@pytest.mark.parametrize("k,na,nb,M,i,nsite", [(8, 4, 4, 64, 3, 1), (9, 4, 4, 60, 4, 2), (10, 2, 2, 131, 4, 1)])
def test_plans_that_share_lists_equal_plans_of_their_own(pkg, k, na, nb, M, i, nsite, kernel):
    """One, two and five vectors in several orders of the calls, every result with the bits of a
    fresh context's own plan; and again after a renormalization dropped the plans."""
    H = synth.ab_initio(k, na, nb, 60 + M)
    want = {}
    x = None
    for nvec in (1, 2, 5):
        c = _context(pkg, H, M, i, nsite, 61, kernel=kernel)
        n, _ = c.wfn_layout(i, nsite)
        if x is None:
            x = torch.tensor(synth.random_vector(5 * n, 62), dtype=torch.float64, device="cuda:0")
            want["d"] = torch.empty(n, dtype=torch.float64, device="cuda:0")
        y = torch.full((nvec * n,), float("nan"), dtype=torch.float64, device="cuda:0")
        c.sigma(i, nsite, x, y, nvec=nvec)
        if nvec == 1:
            c.heff_diag(i, nsite, want["d"])
        torch.cuda.synchronize()
        want[nvec] = y
        c.close()
    for order in ((1, 2, 5), (5, 1, 2), ("d", 5, 1, 2), (2, "d", 5, 1)):
        c = _context(pkg, H, M, i, nsite, 61, kernel=kernel)
        for _ in range(2):
            for what in order:
                y = torch.full_like(want[what], float("nan"))
                if what == "d":
                    c.heff_diag(i, nsite, y)
                else:
                    c.sigma(i, nsite, x, y, nvec=what)
                torch.cuda.synchronize()
                assert torch.equal(y, want[what]), (order, what)
            c.renormalize(i - 1, +1)
        c.close()
