"""FP64 products whose operands span many orders of magnitude (GPU)."""
import numpy as np
import pytest

import synth
from oracle import mps as om

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KERNEL_FP64 = 1   # the FP64 FMA tiles for every list: the reference arithmetic


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_1646_gb300 import build
    build.build()
    import paper_1311_1646_gb300 as p
    p.load()
    return p


def _graded_reference(k, na, nb, M, seed, span):
    """A mixed-canonical MPS whose Schmidt values fall over orders of magnitude: the bonds of a
    random MPS damped by 1 .. 10^-span per sector, then brought to its canonical forms."""
    m = synth.random_mps(k, na, nb, M, seed)
    sites = [om.unpack_site(m.sites[j], m.bonds[j], m.bonds[j + 1]) for j in range(k)]
    for j in range(k - 1):
        sites[j] = {q: A * 10.0 ** (-span * np.arange(A.shape[1]) / max(A.shape[1], 2)) for q, A in sites[j].items()}
    return om.mixed_canonical(sites)


def _tda(pkg, H, ref, n, kernel, **kw):
    L0, R0, C0, Lam, _ = ref
    k = H.k
    tables = [[(q[0], q[1], len(Lam[b][q])) for q in sorted(Lam[b])] for b in range(k + 1)]
    pack = [[om.pack_site(T[i], tables[i], tables[i + 1]) for i in range(k)] for T in (L0, R0, C0)]
    lam = [np.concatenate([Lam[b][q] for q in sorted(Lam[b])]) for b in range(k + 1)]
    ctx = pkg.Context(0)
    ctx.set_kernels(kernel)
    ctx.op_build(k, H.h, H.eri, e_core=H.e_core)
    ctx.mps_load(k, H.n_alpha, H.n_beta, tables, pack[0], 0, sites_right=pack[1])
    ctx.tda_load(pack[2], lam)
    out = ctx.sweep_tda(n, allow_noconv=True, **kw)
    ctx.close()
    return out


@pytest.mark.parametrize("M,span", [(40, 4), (64, 4), (40, 6), (64, 6)])
def test_tda_with_small_schmidt_values_is_as_accurate_as_fma_products(pkg, M, span):
    """One tangent-space sweep after the start sweep, on Schmidt values down to below 1e-6: the
    products with Lambda^-1 magnify every error that is relative to a row's or column's largest
    element only.  Products accurate element by element leave the roots of the two arithmetics
    within about 1e4 roundings of 1e-16 of the energies involved (about 20): 1e-12 * 20 at most."""
    H = synth.ab_initio(8, 4, 4, 5)
    ref = _graded_reference(8, 4, 4, M, 3, span)
    assert min(x.min() for b in range(H.k + 1) for x in ref[3][b].values()) < 1e-6
    w0, r0, e0 = _tda(pkg, H, ref, 2, KERNEL_FP64, max_iter=1, eps=1e-30)
    w1, r1, e1 = _tda(pkg, H, ref, 2, 0, max_iter=1, eps=1e-30)
    assert abs(e1 - e0) <= 1e-12 * abs(e0)
    assert np.abs(w1 - w0).max() <= 1e-12 * abs(e0)
    assert np.abs(r1 / r0 - 1.0).max() <= 1e-12 * abs(e0)
