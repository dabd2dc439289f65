"""The FP32 preconditioner at the launch shapes of large cells: planes of more items than
threads (several rounds per thread), planes close to the shared-memory limit and just above
it, rows that are no whole 16-byte words (the passes take the last two), extents of 512 along
axes 2 and 3, against the FP64 form on the same right-hand sides.

Bound 1e-4, as against the oracle: every iteration rounds sums of 138 terms (about 1e-5
of the operator's norm in the worst case) and a few iterations of a well-conditioned system
amplify that by less than ten."""
import numpy as np
import pytest

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
    ((48, 48, 4), 3, 3),      # 96^2 points: 288 items on 160 threads
    ((64, 40, 3), 2, 3),      # 320 items, two rounds of 160
    ((118, 118, 2), 2, 3),    # 222784 of 225280 bytes
    ((120, 119, 2), 2, 2),    # above the limit: by passes
    ((47, 48, 4), 2, 3),      # rows of 94 points: by passes
    ((4, 256, 3), 2, 3),      # 512 rows, wrapped table of the largest size
    ((2, 3, 256), 2, 3),      # columns of 512 points, 512 threads
    ((40, 44, 256), 1, 2),    # both large
])
def test_against_fp64(W, n, norb, ncg):
    import torch
    g = W.Grid(n, (0.25, 0.3, 0.2))
    G = torch.from_numpy(inputs.orbitals(79, norb, n).astype(np.float32)).cuda()
    eps = torch.linspace(-0.3, -1.1, norb, dtype=torch.float64, device="cuda")
    x, rr = W.precondition(G, eps, g, ncg)
    y, ry = W.precondition(G.double(), eps, g, ncg)
    x, y, g2 = x.double(), y, (G.double() ** 2).sum(1)
    for o in range(norb):
        assert float((x[o] - y[o]).abs().max()) <= 1e-4 * float(y[o].abs().max())
        assert abs(float(rr[o] - ry[o])) <= 1e-3 * float(ry[o]) + 1e-8 * float(g2[o])
