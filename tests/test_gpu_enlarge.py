"""Enlargement of operator sets with device-resolved sources (GPU): environments carried
across the middle bond (where the pair operators turn complementary) from either end, the
sigma at the far side against the oracle.  Block sizes around the kernel's edges: one element,
16 and fewer (references spread over lanes), 32, and more than one work item of 128."""
import numpy as np
import pytest

import synth
from oracle import blocks as ob
from oracle import fock
from oracle import mps as om

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RTOL = 1e-12   # relative to max|y|, the FP64 agreement bar for sigma


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_1646_gb300 import build
    build.build()
    import paper_1311_1646_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("k,na,nb,M", [(6, 1, 0, 2), (7, 3, 4, 16), (8, 4, 4, 70), (8, 2, 2, 160)])
@pytest.mark.parametrize("far", ["left", "right"])
def test_environment_across_the_middle(pkg, k, na, nb, M, far):
    i = k - 2 if far == "left" else 1
    H = synth.ab_initio(k, na, nb, 70 + M)
    m = synth.mixed_mps(k, na, nb, M, 71, center=i)
    ctx = pkg.Context(0)
    ctx.op_build(k, H.h, H.eri)
    ctx.mps_load(k, na, nb, m.bonds, m.sites, i)
    t, v = fock.spin_integrals(H.h, H.eri)
    env = ob.Environment(H, t, v)
    sites = [om.unpack_site(m.sites[j], m.bonds[j], m.bonds[j + 1]) for j in range(k)]
    for b in range(i):
        ctx.renormalize(b, +1)
        env.grow_left(b, sites[b])
    for b in range(k - 1, i, -1):
        ctx.renormalize(b, -1)
        env.grow_right(b, sites[b])
    n, _ = ctx.wfn_layout(i, 1)
    x = synth.random_vector(n, 72)
    xd = torch.tensor(x, dtype=torch.float64, device="cuda:0")
    yd = torch.full_like(xd, float("nan"))
    ctx.sigma(i, 1, xd, yd)
    y = yd.cpu().numpy()
    ref = om.pack_site(ob.sigma_onesite(env, i, om.unpack_site(x, m.bonds[i], m.bonds[i + 1])), m.bonds[i], m.bonds[i + 1])
    assert np.abs(y - ref).max() <= RTOL * np.abs(ref).max()
    ctx.close()
