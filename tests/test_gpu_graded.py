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


@pytest.mark.parametrize("kernel", [0, 2, 3])
@pytest.mark.parametrize("M,span", [(40, 4), (64, 4), (40, 6), (64, 6)])
def test_tda_with_small_schmidt_values_is_as_accurate_as_fma_products(pkg, M, span, kernel):
    """One tangent-space sweep after the start sweep, on Schmidt values down to below 1e-6: the
    products with Lambda^-1 magnify every error that is relative to a row's or column's largest
    element only.  Products accurate element by element leave the roots of the two arithmetics
    within about 1e4 roundings of 1e-16 of the energies involved (about 20): 1e-12 * 20 at most."""
    H = synth.ab_initio(8, 4, 4, 5)
    ref = _graded_reference(8, 4, 4, M, 3, span)
    assert min(x.min() for b in range(H.k + 1) for x in ref[3][b].values()) < 1e-6
    w0, r0, e0 = _tda(pkg, H, ref, 2, KERNEL_FP64, max_iter=1, eps=1e-30)
    w1, r1, e1 = _tda(pkg, H, ref, 2, kernel, max_iter=1, eps=1e-30)
    assert abs(e1 - e0) <= 1e-12 * abs(e0)
    assert np.abs(w1 - w0).max() <= 1e-12 * abs(e0)
    assert np.abs(r1 / r0 - 1.0).max() <= 1e-12 * abs(e0)


def _scaled_gauge(m, k, i, nsite, side, span, seed):
    """The MPS with every state of the left (right) bases scaled by its own power of two, 1 to
    2^-span: the renormalized operators of that side scale by row and column, exactly."""
    rng = np.random.default_rng(seed)
    S = []
    for b, table in enumerate(m.bonds):
        on = 0 < b <= i if side == "left" else i + nsite <= b < k
        S.append({(qa, qb): 2.0 ** -(rng.integers(0, span + 1, size=d) if on else np.zeros(d)) for qa, qb, d in table})
    sites = []
    for j in range(k):
        A = om.unpack_site(m.sites[j], m.bonds[j], m.bonds[j + 1])
        if j < i:
            A = {q: X / S[j][q[0]][:, None] * S[j + 1][q[2]][None, :] for q, X in A.items()}
        elif j >= i + nsite:
            A = {q: X * S[j][q[0]][:, None] / S[j + 1][q[2]][None, :] for q, X in A.items()}
        sites.append(om.pack_site(A, m.bonds[j], m.bonds[j + 1]))
    return S, sites


def _wave_scale(m, S, i, nsite, n):
    b = m.bonds
    if nsite == 1:
        w = {q: X * S[i][q[0]][:, None] * S[i + 1][q[-1]][None, :]
             for q, X in om.unpack_site(np.ones(n), b[i], b[i + 1]).items()}
        return om.pack_site(w, b[i], b[i + 1])
    w = {q: X * S[i][q[0]][:, None] * S[i + 2][q[-1]][None, :]
         for q, X in om.unpack_twosite(np.ones(n), b[i], b[i + 2]).items()}
    return om.pack_twosite(w, b[i], b[i + 2])


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("side", ["left", "right"])
@pytest.mark.parametrize("k,na,nb,M,i,nsite", [(10, 2, 2, 131, 4, 1), (9, 4, 4, 60, 4, 2)])
def test_sigma_in_a_graded_gauge(pkg, k, na, nb, M, i, nsite, side, kernel):
    """Basis states scaled by 2^0 to 2^-30 and the vector by the inverse: along K one operand rises
    as the other falls, by 2^60 on the two-sided operators.  Against the FMA tiles on the same
    input, relative to the largest element, at the bar of every FP64 sigma; and several vectors
    in one call give each vector's own bits."""
    H = synth.ab_initio(k, na, nb, 7)
    m = synth.mixed_mps(k, na, nb, M, 8, center=i)
    S, sites = _scaled_gauge(m, k, i, nsite, side, 30, 1)
    out = []
    for kn in (KERNEL_FP64, kernel):
        ctx = pkg.Context(0)
        ctx.set_kernels(kn)
        ctx.op_build(k, H.h, H.eri)
        ctx.mps_load(k, na, nb, m.bonds, sites, i)
        for b in range(i):
            ctx.renormalize(b, +1)
        for b in range(k - 1, i + nsite - 1, -1):
            ctx.renormalize(b, -1)
        n, _ = ctx.wfn_layout(i, nsite)
        x = synth.random_vector(2 * n, 9) / np.tile(_wave_scale(m, S, i, nsite, n), 2)
        xd = torch.tensor(x, dtype=torch.float64, device="cuda:0")
        y, y1 = torch.empty_like(xd), torch.empty_like(xd)
        ctx.sigma(i, nsite, xd, y, nvec=2)
        ctx.sigma(i, nsite, xd[:n], y1[:n])
        ctx.sigma(i, nsite, xd[n:], y1[n:])
        torch.cuda.synchronize()
        assert torch.equal(y, y1)
        out.append(y.cpu().numpy())
        ctx.close()
    assert np.abs(out[1] - out[0]).max() <= 1e-12 * np.abs(out[0]).max()


@pytest.mark.parametrize("kernel", [2, 3])
def test_subnormal_vectors_are_multiplied(pkg, kernel):
    """A vector of subnormals only (46 bits and fewer) under a Hamiltonian of exponent 2^400: the
    result is a normal number of about 40 bits, as from the FMA tiles (1e-11: the rounding of
    subnormal intermediates to multiples of 2^-1074, a few of 2^-46 each)."""
    k, na, nb, M, i = 10, 2, 2, 60, 4
    H = synth.ab_initio(k, na, nb, 7)
    m = synth.mixed_mps(k, na, nb, M, 8, center=i)
    out = []
    for kn in (KERNEL_FP64, kernel):
        ctx = pkg.Context(0)
        ctx.set_kernels(kn)
        ctx.op_build(k, H.h * 2.0 ** 400, H.eri * 2.0 ** 400)
        ctx.mps_load(k, na, nb, m.bonds, m.sites, i)
        for b in range(i):
            ctx.renormalize(b, +1)
        for b in range(k - 1, i, -1):
            ctx.renormalize(b, -1)
        n, _ = ctx.wfn_layout(i, 1)
        x = synth.random_vector(2 * n, 9)
        x[:n] = np.round(x[:n] / np.abs(x[:n]).max() * 2.0 ** 46) * 2.0 ** -1000 * 2.0 ** -74
        assert np.abs(x[:n]).max() < 2.0 ** -1022 and np.any(x[:n] != 0.0)
        xd = torch.tensor(x, dtype=torch.float64, device="cuda:0")
        y = torch.empty_like(xd)
        ctx.sigma(i, 1, xd, y, nvec=2)
        torch.cuda.synchronize()
        out.append(y.cpu().numpy())
        ctx.close()
    for v in (slice(0, n), slice(n, 2 * n)):
        assert np.abs(out[0][v]).max() > 0.0
        assert np.abs(out[1][v] - out[0][v]).max() <= (1e-11 if v.start == 0 else 1e-12) * np.abs(out[0][v]).max()
