"""The FP32 passes by transposed tiles at the edges of their tiles, with as many orbitals as
send a call of such cells there (5e5 points): rows shorter than, equal to and not a multiple
of the half tile, lines of less than a chunk, of exactly one and of several per thread, planes
of an odd number of coarse points (every word width), groups of orbitals with a density; H psi,
both energies and the density against the oracle, and the same bits as the row-wise kernels
that a few orbitals take.

Bounds, normwise, of the other FP32 passes: 2e-6, 5e-6 for the density (the square); 1e-6
for the energies (terms accurate to a few 1e-7, summed in FP64)."""
import numpy as np
import pytest

import oracle.wavelet as O
from paper_0904_1543_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL, TOL_RHO, TOL_E = 2e-6, 5e-6, 1e-6
NDIST = 5   # orbitals that differ; a call repeats them


@pytest.fixture(scope="module")
def W():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0904_1543_gb300 as W
    return W


def cuda(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def err(got, ref):
    return np.abs(got.detach().double().cpu().numpy().reshape(ref.shape) - ref).max() / np.abs(ref).max()


SIZES = [(1, 1, 1), (3, 5, 2), (7, 9, 5), (33, 2, 4), (5, 17, 2), (3, 2, 17), (9, 5, 16), (7, 3, 31), (20, 29, 13),
         (300, 2, 3), (3, 2, 260)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("density", [False, True])
def test_large_calls(W, n, density):
    import torch
    g = W.Grid(n, (0.25, 0.3, 0.2))
    norb = 500000 // g.ncoef + 3
    base = inputs.orbitals(191, NDIST, n).astype(np.float32)
    V = inputs.gaussian_potential(191, 0, n).astype(np.float32)
    which = np.arange(norb) % NDIST
    occ = 0.5 + (np.arange(norb) % 3) / 2.0
    psi = cuda(base)[cuda(which)]
    rho = torch.full(g.fine, 0.25, dtype=torch.float64, device="cuda") if density else None
    hp, ek, ep = W.hpsi_local(psi, cuda(V), cuda(occ), g, rho=rho)
    hr, _, ekr, epr = O.hpsi_batch(base.astype(np.float64), V.astype(np.float64), np.ones(NDIST), n, (0.25, 0.3, 0.2))
    pick = sorted({0, 1, norb // 2, norb - 2, norb - 1})
    w = which[pick]
    assert err(hp[pick], hr.reshape(NDIST, -1)[w]) <= TOL
    assert np.all(np.abs(ek.cpu().numpy()[pick] - ekr[w]) <= TOL_E * np.abs(ekr[w]))
    assert np.all(np.abs(ep.cpu().numpy()[pick] - epr[w]) <= TOL_E * np.abs(epr[w]))
    # every repetition of an orbital is the same, and a small call's
    for k in range(NDIST):
        assert torch.equal(hp[k::NDIST], hp[k:k + 1].expand_as(hp[k::NDIST]))
    few = W.hpsi_local(psi[:NDIST], cuda(V), cuda(occ[:NDIST]), g)
    assert torch.equal(few[0], hp[:NDIST])
    if density:
        share = np.array([occ[which == k].sum() for k in range(NDIST)])
        ref = sum(share[k] * O.density(base[k].astype(np.float64), 1.0, n) for k in range(NDIST))
        assert err(rho - 0.25, ref) <= TOL_RHO


@pytest.mark.parametrize("n", SIZES)
def test_large_operators(W, n):
    import torch
    g = W.Grid(n)
    norb = 500000 // g.ncoef + 2
    x = inputs.random_field(192, 0, (NDIST,) + g.fine).astype(np.float32)
    x.reshape(NDIST, -1)[0, :3] = [1e3, -1e3, 1e3]
    idx = cuda(np.arange(norb) % NDIST)
    big = cuda(x)[idx]
    syn = W.synthesis(big.reshape(norb, -1), g)
    ana = W.analysis(big, g)
    for k in range(NDIST):
        c = x[k].astype(np.float64)
        last = norb - 1 - (norb - 1 - k) % NDIST
        for o in {k, last}:
            assert err(syn[o], O.synthesis3d(O.uncompress(c.reshape(-1), n))) <= TOL
            assert err(ana[o], O.compress(O.analysis3d(c), n)) <= TOL
    few = cuda(x)
    assert torch.equal(W.synthesis(few.reshape(NDIST, -1), g), syn[:NDIST])
    assert torch.equal(W.analysis(few, g), ana[:NDIST])
