"""FP32 boxes with one to three free axes on both sides of the potential pass's rule
(small calls by rows, large ones by transposed tiles), several orbitals per density
group, with and without a density, every result against the free-space oracle.

Bounds, normwise, as for the periodic passes: fifteen passes of at most 29 products of
relative error 2^-24 with gains below 2 stay within a few 1e-7 unless the roundings
conspire: 2e-6, 5e-6 for the density (the square), 1e-6 for the energies (of terms
accurate to the same few 1e-7, summed in FP64)."""
import numpy as np
import pytest

import oracle.free as FR
from paper_0904_1543_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL, TOL_RHO, TOL_E = 2e-6, 5e-6, 1e-6
NDIST = 3   # orbitals that differ; a call repeats them with other occupations


@pytest.fixture(scope="module")
def W():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0904_1543_gb300 as W
    return W


# axis 3 has 32 or more output lines' points, so that calls with a density reach both forms
CASES = [((1, 1, 1), (6, 5, 7), (2, 20)), ((0, 1, 0), (4, 6, 17), (3, 50)), ((1, 0, 0), (6, 4, 17), (1, 50)),
         ((1, 1, 0), (5, 4, 16), (4, 13)), ((0, 0, 1), (5, 7, 3), (2, 300))]


@pytest.mark.parametrize("free,n,counts", CASES)
@pytest.mark.parametrize("density", [False, True])
def test_free_axes(W, free, n, counts, density):
    import torch
    g = W.Grid(n, (0.25, 0.3, 0.2))
    pad = W.FREE_PAD
    padded = tuple(v + (2 * pad if free[d] else 0) for d, v in enumerate(n))
    base = inputs.orbitals(117, NDIST, n).astype(np.float32)
    V = inputs.gaussian_potential(117, 0, padded).astype(np.float32)
    Vx = FR.extend_bc(V.astype(np.float64), n, 2 * pad, free)
    refs = [FR.hpsi_local_bc(base[k].astype(np.float64), Vx, 1.0, n, free, g.h) for k in range(NDIST)]
    for norb in counts:
        which = np.arange(norb) % NDIST
        occ = 0.5 + (np.arange(norb) % 4) / 2.0
        rho = torch.zeros(W.bc_fine(g, free), dtype=torch.float64, device="cuda") if density else None
        hp, ek, ep = W.hpsi_local_bc(torch.from_numpy(base[which]).cuda(), torch.from_numpy(V).cuda(),
                                     torch.from_numpy(occ).cuda(), g, free, rho=rho)
        hp, ek, ep = hp.double().cpu().numpy(), ek.cpu().numpy(), ep.cpu().numpy()
        ref_rho = 0.0
        for o in range(norb):
            r = refs[which[o]]
            h = r["hpsi_c"]
            assert np.abs(hp[o].reshape(h.shape) - h).max() <= TOL * np.abs(h).max()
            assert abs(ek[o] - r["ekin"]) <= TOL_E * abs(r["ekin"])
            assert abs(ep[o] - r["epot"]) <= TOL_E * abs(r["epot"])
            ref_rho = ref_rho + occ[o] * r["rho"]
        if density:
            ref = FR.restrict_bc(ref_rho, n, 2 * pad, free)
            assert np.abs(rho.cpu().numpy() - ref).max() <= TOL_RHO * np.abs(ref).max()
