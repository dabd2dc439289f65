"""The FP32 compressed and potential passes at the edges of their tiles: rows shorter
than, equal to and not a multiple of the half tile, lines of less than one chunk, of several
chunks per thread (their results go behind the tile), planes of an odd number of coarse
points (every word width), orbital groups with and without a density, against the
oracle on the FP32-rounded inputs.

Bounds, normwise: a pass sums at most 16 products (29 in the kinetic passes), each
rounded to 2^-24; three passes per operator, fifteen in H psi, with every gain below 2, leave below
15 x 29 x 2^-24 = 2.6e-5 in the worst case and a few 1e-7 when the roundings do not
conspire: 2e-6, and 5e-6 for the density, the square."""
import numpy as np
import pytest

import oracle.wavelet as O
from paper_0904_1543_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL, TOL_RHO = 2e-6, 5e-6


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


SIZES = [((1, 1, 1), 3), ((2, 1, 3), 5), ((3, 5, 2), 700), ((4, 4, 4), 2), ((7, 9, 5), 40), ((8, 3, 8), 130),
         ((16, 17, 2), 60), ((33, 2, 4), 30), ((5, 6, 61), 90), ((20, 30, 130), 4), ((300, 2, 3), 60)]


@pytest.mark.parametrize("n,norb", SIZES)
def test_operators(W, n, norb):
    g = W.Grid(n)
    x = inputs.random_field(91, 0, (norb,) + g.fine).astype(np.float32)
    x.reshape(norb, -1)[0, :3] = [1e3, -1e3, 1e3]   # a large entry at the first points
    syn = W.synthesis(cuda(x.reshape(norb, -1)), g)
    ana = W.analysis(cuda(x), g)
    for o in {0, norb // 2, norb - 1}:
        c = x[o].astype(np.float64)
        assert err(syn[o], O.synthesis3d(O.uncompress(c.reshape(-1), n))) <= TOL
        assert err(ana[o], O.compress(O.analysis3d(c), n)) <= TOL


@pytest.mark.parametrize("n,norb", SIZES)
@pytest.mark.parametrize("density", [False, True])
def test_hpsi(W, n, norb, density):
    import torch
    g = W.Grid(n)
    norb = min(norb, 130)
    psi = inputs.orbitals(92, norb, n).astype(np.float32)
    V = inputs.gaussian_potential(92, 0, n).astype(np.float32)
    occ = np.linspace(2.0, 0.0, norb)
    rho = torch.full(g.fine, 0.25, dtype=torch.float64, device="cuda") if density else None
    hp, _, _ = W.hpsi_local(cuda(psi), cuda(V), cuda(occ), g, rho=rho)
    psi64, V64 = psi.astype(np.float64), V.astype(np.float64)
    if density:
        hr, rr, _, _ = O.hpsi_batch(psi64, V64, occ, n)
        assert err(hp, hr) <= TOL
        assert err(rho - 0.25, rr) <= TOL_RHO
    else:
        pick = sorted({0, norb // 2, norb - 1})
        hr, _, _, _ = O.hpsi_batch(psi64[pick], V64, occ[pick], n)
        assert err(hp[pick], hr) <= TOL


@pytest.mark.parametrize("n,norb", [((3, 5, 2), 7), ((8, 3, 9), 40), ((12, 13, 14), 20)])
def test_same_as_row_wise(W, n, norb):
    """A region that holds every point takes the row-wise kernel for the compressed
    passes: the same sums in the same order."""
    import torch
    g = W.Grid(n)
    reg = W.Region(g, np.ones(n[::-1], bool), np.ones(n[::-1], bool), bounds=False)
    psi = cuda(inputs.orbitals(93, norb, n).astype(np.float32))
    V = cuda(inputs.gaussian_potential(93, 0, n).astype(np.float32))
    occ = cuda(np.full(norb, 2.0))
    a = W.hpsi_local(psi, V, occ, g)
    b = W.hpsi_local_region(psi, V, occ, g, reg)
    assert torch.equal(a[0], b[0])
    for x, y in zip(a[1:], b[1:]):
        assert torch.allclose(x, y, rtol=1e-12)
