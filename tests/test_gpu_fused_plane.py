"""The transposing plane kernels of the FP32 fused chain: every square plane they take
(32 to 128 points a side), with a density, without one, for the density and for the
energies alone, several cells (of one launch and of the general form) in a plan, and
more planes than two per SM, where they run; against the oracle, and against the general
form, which a plan of few planes takes.

Bounds, normwise: the FP32 bounds of the fused chain (H psi 2e-6, density 5e-6,
energies 5e-7 relative, on cells of at least 8192 points).  Against the general form: t, the
density and the energies' chains keep its order (the same bits, the energies' outer sums to
1e-12); H psi differs by the rounding of two exchanged 16-tap filters, 2 x 16 x 2^-24 = 1.9e-6
of the largest value."""
import numpy as np
import pytest

import oracle.wavelet as O
from paper_0904_1543_gb300 import inputs

pytestmark = pytest.mark.gpu


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
    got, ref = (x.detach().double().cpu().numpy() if hasattr(x, "detach") else np.asarray(x) for x in (got, ref))
    return np.abs(got.reshape(ref.shape) - ref).max() / np.abs(ref).max()


def run(W, grids, cells, psi, V, occ, density=True):
    import torch
    plan = W.Plan(grids, cells, prec=W.WVL_F32, graph=False, chain="fused")
    rho = [torch.zeros(g.fine, dtype=torch.float64, device="cuda") for g in grids] if density else None
    hp = torch.empty_like(psi)
    ek = torch.empty(len(cells), dtype=torch.float64, device="cuda")
    ep = torch.empty_like(ek)
    plan.hpsi(psi, V, occ, hpsi=hp, rho=rho, ekin=ek, epot=ep)
    return hp, rho, ek, ep


@pytest.mark.parametrize("n", [(16, 16, 20), (32, 32, 16), (48, 48, 20), (64, 64, 16)])
@pytest.mark.parametrize("density", [False, True])
def test_square_planes(W, n, density):
    import torch
    g = W.Grid(n)
    norb = 320 // (2 * n[2]) + 2
    assert norb * 2 * n[2] > 2 * 152
    psi = inputs.orbitals(97, norb, n).astype(np.float32)
    V = inputs.gaussian_potential(97, 0, n).astype(np.float32)
    occ = np.linspace(2.0, 1.0, norb)
    hp, rho, ek, ep = run(W, [g], [0] * norb, cuda(psi.reshape(-1)), [cuda(V)], cuda(occ), density)
    hp = hp.reshape(norb, -1)
    pick = [0, norb // 2, norb - 1]
    hr, _, ekr, epr = O.hpsi_batch(psi[pick].astype(np.float64), V.astype(np.float64), occ[pick], n)
    assert err(hp[pick], hr) <= 2e-6
    assert np.all(np.abs(ek.cpu().numpy()[pick] - ekr) <= 5e-7 * np.abs(ekr))
    assert np.all(np.abs(ep.cpu().numpy()[pick] - epr) <= 5e-7 * np.abs(epr))
    # few orbitals per call: the general form
    m = max(1, 304 // (2 * n[2]))
    gho = torch.zeros(g.fine, dtype=torch.float64, device="cuda")
    for o in range(0, norb, m):
        q = slice(o, min(norb, o + m))
        k = q.stop - o
        h2, r2, k2, p2 = run(W, [g], [0] * k, cuda(psi[q].reshape(-1)), [cuda(V)], cuda(occ[q]), density)
        assert err(hp[q], h2.reshape(k, -1)) <= 1.9e-6
        assert torch.allclose(ek[q], k2, rtol=1e-12) and torch.allclose(ep[q], p2, rtol=1e-12)
        if density:
            gho += r2[0]
    if density:
        assert torch.allclose(rho[0], gho, rtol=1e-12, atol=0.0)


def test_cells_of_both_forms(W):
    import torch
    sizes = [(16, 16, 20), (16, 20, 16), (32, 32, 16), (16, 16, 16)]
    grids = [W.Grid(n) for n in sizes]
    cells = [0] * 10 + [1] * 12 + [2] * 11 + [3] * 12
    parts = [inputs.orbitals(98 + k, cells.count(k), n).astype(np.float32) for k, n in enumerate(sizes)]
    V = [inputs.gaussian_potential(98, k, n).astype(np.float32) for k, n in enumerate(sizes)]
    occ = np.linspace(1.0, 2.0, len(cells))
    psi = np.concatenate([p.reshape(-1) for p in parts])
    hp, rho, ek, ep = run(W, grids, cells, cuda(psi), [cuda(v) for v in V], cuda(occ))
    at, o = 0, 0
    for k, n in enumerate(sizes):
        m = parts[k].size
        hr, rr, ekr, epr = O.hpsi_batch(parts[k].astype(np.float64), V[k].astype(np.float64),
                                        occ[o:o + len(parts[k])], n)
        assert err(hp[at:at + m], hr) <= 2e-6 and err(rho[k], rr) <= 5e-6
        assert np.all(np.abs(ek.cpu().numpy()[o:o + len(parts[k])] - ekr) <= 5e-7 * np.abs(ekr))
        at += m
        o += len(parts[k])


@pytest.mark.parametrize("n", [16, 64])
def test_density_and_energies_alone(W, n):
    """The chain without v: energies without H psi, the density without either."""
    import torch
    n = (n, n, 16)
    g = W.Grid(n)
    norb = 12
    psi = inputs.orbitals(99, norb, n).astype(np.float32)
    V = inputs.gaussian_potential(99, 0, n).astype(np.float32)
    occ = np.linspace(2.0, 0.5, norb)
    rho = W.density(cuda(psi), cuda(occ), g)
    ek, ep = W.energy(cuda(psi), cuda(V), cuda(occ), g)[:2]
    _, rr, ekr, epr = O.hpsi_batch(psi.astype(np.float64), V.astype(np.float64), occ, n)
    assert err(rho, rr) <= 5e-6
    assert np.all(np.abs(ek.cpu().numpy() - ekr) <= 5e-7 * np.abs(ekr))
    assert np.all(np.abs(ep.cpu().numpy() - epr) <= 5e-7 * np.abs(epr))
