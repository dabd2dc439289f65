"""The FP32 preconditioner by the separable operator at the edges of its kernels:
extents below, at and above the 46-tap filter and the 8-row items, partial
tiles of 32 columns, one and several orbitals, one to several iterations, against the
oracle; the kernels that other extents take agree with it.

Bound 1e-4: every iteration rounds sums of 138 terms (about 1e-5 of the operator's
norm in the worst case) and a few iterations of a well-conditioned system
amplify that by less than ten."""
import numpy as np
import pytest

import oracle.precond as PC
from paper_0904_1543_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0904_1543_gb300 as W
    return W


@pytest.mark.parametrize("n,norb,ncg", [
    ((2, 1, 1), 2, 1), ((2, 3, 2), 1, 2), ((4, 4, 13), 3, 3), ((6, 11, 5), 2, 4), ((22, 4, 12), 2, 1),
    ((24, 9, 23), 1, 3), ((12, 13, 14), 3, 5), ((3, 4, 6), 2, 3)])
@pytest.mark.parametrize("residual", [False, True])
def test_against_oracle(W, n, norb, ncg, residual):
    import torch
    h = (0.25, 0.3, 0.2)
    G = inputs.orbitals(76, norb, n).astype(np.float32)
    eps = np.linspace(-0.3, -1.1, norb)
    g = torch.from_numpy(G).cuda()
    x, rr = W.precondition(g, torch.from_numpy(eps).cuda(), W.Grid(n, h), ncg, want_residual=residual)
    x = x.double().cpu().numpy()
    for o in range(norb):
        ref = PC.precondition(G[o].astype(np.float64), eps[o], n, ncg, h)
        assert np.abs(x[o] - ref).max() <= 1e-4 * np.abs(ref).max()
        if residual:
            res = G[o].astype(np.float64) - PC.helmholtz_apply(ref, eps[o], n, h)
            assert abs(float(rr[o]) - res @ res) <= 1e-3 * (res @ res) + 1e-8 * (G[o] @ G[o])
    assert torch.equal(g.cpu(), torch.from_numpy(G))


def test_small_values(W):
    """Right-hand sides whose products leave the range of FP32: the scalars are then
    formed in FP64, and x scales with g."""
    import torch
    n = (8, 6, 7)
    G = inputs.orbitals(77, 2, n).astype(np.float32)
    eps = torch.tensor([-0.4, -0.9], dtype=torch.float64, device="cuda")
    x, _ = W.precondition(torch.from_numpy(G).cuda(), eps, W.Grid(n), 3)
    s = np.float32(2.0 ** -70)
    y, _ = W.precondition(torch.from_numpy(G * s).cuda(), eps, W.Grid(n), 3)
    x, y = x.double().cpu().numpy(), y.double().cpu().numpy() * 2.0 ** 70
    assert np.abs(x - y).max() <= 1e-5 * np.abs(x).max()
