"""The FP64 grouped GEMM as exact digit products on the tensor cores (GPU): sectors wide
enough that the plans take that kernel (work padded to 16 x 8 x 16 at most 3 times the exact
work), at tile and chunk edges, against the oracle; and the exponent range beyond which its
chunks are multiplied in plain FP64."""
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


def _context(pkg, k, na, nb, M, i, nsite, h, eri, m):
    ctx = pkg.Context(0)
    ctx.op_build(k, h, eri)
    ctx.mps_load(k, na, nb, m.bonds, m.sites, i)
    for b in range(i):
        ctx.renormalize(b, +1)
    for b in range(k - 1, i + nsite - 1, -1):
        ctx.renormalize(b, -1)
    return ctx


def _sigma(pkg, ctx, i, nsite, x, nvec):
    xd = torch.tensor(x, dtype=torch.float64, device="cuda:0")
    yd = torch.full_like(xd, float("nan"))
    ctx.sigma(i, nsite, xd, yd, nvec=nvec)
    torch.cuda.synchronize()
    return yd.cpu().numpy()


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


# few electrons in many orbitals: sectors of 16 to 66 states, sub-blocks just below, at and
# above the tiles' 16s, chunks of 32 positions that hold one or several segments
@pytest.mark.parametrize("k,na,nb,M,i,nsite,nvec", [
    (8, 1, 1, 16, 3, 1, 1), (8, 1, 1, 17, 3, 1, 2), (10, 2, 1, 60, 4, 1, 3), (9, 1, 2, 96, 4, 2, 1),
    (10, 2, 2, 131, 4, 1, 5), (10, 2, 2, 190, 5, 2, 2)])
def test_wide_sectors_match_the_oracle(pkg, k, na, nb, M, i, nsite, nvec):
    H = synth.ab_initio(k, na, nb, 60 + M)
    m = synth.mixed_mps(k, na, nb, M, 61, center=i)
    ctx = _context(pkg, k, na, nb, M, i, nsite, H.h, H.eri, m)
    n, _ = ctx.wfn_layout(i, nsite)
    x = synth.random_vector(nvec * n, 62)
    y = _sigma(pkg, ctx, i, nsite, x, nvec)
    ref = _oracle(H, m, i, nsite)
    for v in range(nvec):
        r = ref(x[v * n:(v + 1) * n])
        assert np.abs(y[v * n:(v + 1) * n] - r).max() <= RTOL * np.abs(r).max(), v
        # a vector's bits do not depend on the others in the call
        assert np.array_equal(_sigma(pkg, ctx, i, nsite, x[v * n:(v + 1) * n], 1), y[v * n:(v + 1) * n])
    ctx.close()


def test_extreme_exponents_and_infinities(pkg):
    """H scaled by 2^-500 puts the operators' exponents outside the integer path's range, so
    the same products run in plain FP64: equal after rescaling, to the rounding of either
    (sums of a few thousand terms: 1e-13).  An infinity in one vector reaches its own result
    only."""
    k, na, nb, M, i = 10, 2, 2, 131, 4
    H = synth.ab_initio(k, na, nb, 7)
    m = synth.mixed_mps(k, na, nb, M, 8, center=i)
    a = _context(pkg, k, na, nb, M, i, 1, H.h, H.eri, m)
    n, _ = a.wfn_layout(i, 1)
    x = synth.random_vector(2 * n, 9)
    y = _sigma(pkg, a, i, 1, x, 2)
    s = 2.0 ** -500
    b = _context(pkg, k, na, nb, M, i, 1, H.h * s, H.eri * s, m)
    z = _sigma(pkg, b, i, 1, x, 2) / s
    assert np.abs(z - y).max() <= 1e-13 * np.abs(y).max()
    x[n // 2] = np.inf
    w = _sigma(pkg, a, i, 1, x, 2)
    assert not np.all(np.isfinite(w[:n]))
    assert np.array_equal(w[n:], y[n:])
    a.close()
    b.close()


# blocks of 1 to 49 states: lanes with one and two elements, digit tiles in both orientations,
# segment lists of one part and of many (their parts added by the last warp), and the CTA tiles
@pytest.mark.parametrize("k,na,nb,M,i,nsite,nvec", [
    (12, 1, 1, 3, 5, 1, 1), (9, 5, 4, 24, 4, 1, 7), (9, 4, 4, 60, 4, 2, 1), (8, 4, 4, 90, 3, 1, 4), (14, 2, 2, 140, 6, 1, 3)])
def test_small_blocks_match_the_oracle(pkg, k, na, nb, M, i, nsite, nvec):
    H = synth.ab_initio(k, na, nb, 90 + M)
    m = synth.mixed_mps(k, na, nb, M, 91, center=i)
    ctx = _context(pkg, k, na, nb, M, i, nsite, H.h, H.eri, m)
    n, _ = ctx.wfn_layout(i, nsite)
    x = synth.random_vector(nvec * n, 92)
    y = _sigma(pkg, ctx, i, nsite, x, nvec)
    ref = _oracle(H, m, i, nsite)
    for v in (0, nvec - 1):
        r = ref(x[v * n:(v + 1) * n])
        assert np.abs(y[v * n:(v + 1) * n] - r).max() <= RTOL * np.abs(r).max(), v
        assert np.array_equal(_sigma(pkg, ctx, i, nsite, x[v * n:(v + 1) * n], 1), y[v * n:(v + 1) * n])
    # the parts' counters are back at zero: the same call again, the same bits
    assert np.array_equal(_sigma(pkg, ctx, i, nsite, x, nvec), y)
    ctx.close()


@pytest.mark.parametrize("first_nvec", [0, 3])
def test_noalloc_single_vector_after_heff_diag(pkg, first_nvec):
    """heff_diag answers from a plan of the diagonal alone or of another vector count; a
    single-vector sigma_noalloc after it gives sigma()'s bits, one of 2 vectors is refused."""
    cfg = synth.config(1)
    H = cfg["ham"]
    m = synth.mixed_mps(H.k, H.n_alpha, H.n_beta, cfg["M"], 77, center=3)
    ctx = _context(pkg, H.k, H.n_alpha, H.n_beta, cfg["M"], 3, 1, H.h, H.eri, m)
    n, _ = ctx.wfn_layout(3, 1)
    if first_nvec:
        _sigma(pkg, ctx, 3, 1, synth.random_vector(first_nvec * n, 4), first_nvec)
    d = torch.empty(n, dtype=torch.float64, device="cuda:0")
    ctx.heff_diag(3, 1, d)
    x = synth.random_vector(2 * n, 5)
    xd = torch.tensor(x, dtype=torch.float64, device="cuda:0")
    yd = torch.full_like(xd, float("nan"))
    with pytest.raises(pkg.LrtError, match="-6"):
        ctx.sigma_noalloc(3, 1, xd, yd, nvec=2)
    ctx.sigma_noalloc(3, 1, xd[:n], yd[:n])
    torch.cuda.synchronize()
    assert np.array_equal(yd[:n].cpu().numpy(), _sigma(pkg, ctx, 3, 1, x[:n], 1))
    ctx.close()
