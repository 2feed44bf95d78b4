"""sigma_batched checks every instance before it does any work (GPU)."""
import ctypes

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


@pytest.mark.parametrize("precision", [0, 1])
def test_a_refused_batch_leaves_the_contexts_untouched(pkg, precision):
    """A NULL vector of the last instance refuses the call; the first instance's operators are
    not enlarged or planned for it (no device memory is taken)."""
    cfg = synth.config(1)
    H = cfg["ham"]
    i = 3
    ctxs, vecs = [], []
    for j in range(2):
        m = synth.mixed_mps(H.k, H.n_alpha, H.n_beta, cfg["M"], 50 + j, center=i)
        c = pkg.Context(0)
        c.op_build(H.k, H.h, H.eri, e_core=H.e_core)
        c.mps_load(H.k, H.n_alpha, H.n_beta, m.bonds, m.sites, i)
        for b in range(i):
            c.renormalize(b, +1)
        for b in range(H.k - 1, i, -1):
            c.renormalize(b, -1)
        n, _ = c.wfn_layout(i, 1)
        ctxs.append(c)
        vecs.append((torch.zeros(n, dtype=torch.float64, device="cuda:0"), torch.zeros(n, dtype=torch.float64, device="cuda:0")))
    vp = ctypes.c_void_p
    hs = (vp * 2)(*[c.h.value for c in ctxs])
    sites = (ctypes.c_int * 2)(i, i)
    px = (vp * 2)(vecs[0][0].data_ptr(), None)
    py = (vp * 2)(*[y.data_ptr() for _, y in vecs])
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    assert ctxs[0].lib.sigma_batched(hs, 2, sites, 1, 1, px, py, precision) == -1
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert free1 == free0
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("nsite", [1, 2])
@pytest.mark.parametrize("kernels", [(1, 2, 3), (3, 0, 2), (2, 2, 2), (0, 0, 0)])
def test_an_instance_of_a_batch_has_the_bits_of_its_own_call(pkg, kernels, nsite):
    """Whatever the other molecules are: each instance keeps its own kernel and K parts, on long
    segment lists (split) and short ones, through the first call and the replayed graph."""
    ctxs, xs, ys, want, sites = [], [], [], [], []
    for j, (k, na, nb, M) in enumerate([(8, 4, 4, 64), (10, 2, 2, 131), (9, 4, 4, 60)]):
        H = synth.ab_initio(k, na, nb, 70 + j)
        i = k // 2 - 1
        m = synth.mixed_mps(k, na, nb, M, 71 + j, center=i)
        c = pkg.Context(0)
        c.set_kernels(kernels[j])
        c.op_build(k, H.h, H.eri)
        c.mps_load(k, na, nb, m.bonds, m.sites, i)
        for b in range(i):
            c.renormalize(b, +1)
        for b in range(k - 1, i + nsite - 1, -1):
            c.renormalize(b, -1)
        n, _ = c.wfn_layout(i, nsite)
        xs.append(torch.tensor(synth.random_vector(3 * n, 72 + j), dtype=torch.float64, device="cuda:0"))
        ys.append(torch.empty_like(xs[-1]))
        want.append(torch.empty_like(xs[-1]))
        c.sigma(i, nsite, xs[-1], want[-1], nvec=3)
        ctxs.append(c)
        sites.append(i)
    for _ in range(3):
        for y in ys:
            y.fill_(float("nan"))
        pkg.sigma_batched(ctxs, sites, nsite, xs, ys, nvec=3)
        torch.cuda.synchronize()
        for j in range(3):
            assert torch.equal(ys[j], want[j]), j
    for c in ctxs:
        c.close()


def test_precision_of_a_mixed_call_is_the_positions_own(pkg):
    """A position that takes split TF32 and one that does not: each as in its own call, in a batch of
    both and for one vector or several."""
    ctxs, xs, ys, sites, want = [], [], [], [], []
    for j, (k, na, nb, M, i) in enumerate([(8, 4, 4, 64, 3), (11, 3, 3, 300, 5)]):
        H = synth.ab_initio(k, na, nb, 80 + j)
        m = synth.mixed_mps(k, na, nb, M, 81 + j, center=i)
        c = pkg.Context(0)
        c.op_build(k, H.h, H.eri)
        c.mps_load(k, na, nb, m.bonds, m.sites, i)
        for b in range(i):
            c.renormalize(b, +1)
        for b in range(k - 1, i, -1):
            c.renormalize(b, -1)
        n, _ = c.wfn_layout(i, 1)
        x = torch.tensor(synth.random_vector(4 * n, 82 + j), dtype=torch.float64, device="cuda:0")
        y64, y = torch.empty_like(x), torch.empty_like(x)
        c.sigma(i, 1, x, y64, nvec=4)
        for nvec in (1, 4):
            before = c.kernel_launches()
            c.sigma(i, 1, x, y, nvec=nvec, precision=pkg.LRT_MIXED)
            after = c.kernel_launches()
            torch.cuda.synchronize()
            assert (after[3] > before[3]) == (j == 1), (j, nvec)
            assert torch.equal(y[:nvec * n], y64[:nvec * n]) == (j == 0)
        ctxs.append(c)
        xs.append(x)
        ys.append(torch.empty_like(x))
        sites.append(i)
        want.append(y64)
    for _ in range(3):
        pkg.sigma_batched(ctxs, sites, 1, xs, ys, nvec=4, precision=pkg.LRT_MIXED)
        torch.cuda.synchronize()
        assert torch.equal(ys[0], want[0])
        e = (ys[1] - want[1]).abs().max().item()
        assert 0.0 < e <= 1e-5 * want[1].abs().max().item()
    for c in ctxs:
        c.close()
