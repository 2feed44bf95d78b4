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
