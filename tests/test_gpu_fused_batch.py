"""An orbital's results in the FP32 fused chain do not depend on the orbitals that share its
call: the number of planes chooses the form of the plane kernels (the transposing one for
square planes of more than two per SM, threads by planes per SM), and every form keeps the same
order of the filter sums and of the FP32 chains of Ekin; the compensated pairs that add the
chains agree to the last bit on these sizes.  The same bits, H psi and both energies."""
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


# transposing planes, then one of every thread count of the general kernels: 512, 256, 160
# (SKM12), 128, 160 (MFTA12), 128, 96 and 64 threads
@pytest.mark.parametrize("n", [(16, 16, 20), (32, 32, 16), (48, 48, 20), (64, 64, 16),
                               (60, 60, 16), (44, 40, 16), (52, 44, 16), (40, 40, 16), (36, 32, 16), (24, 36, 16),
                               (36, 20, 16), (24, 24, 20), (20, 16, 20), (16, 20, 16)])
def test_same_bits(W, n):
    import torch
    g = W.Grid(n, (0.25, 0.3, 0.2))
    norb = 320 // (2 * n[2]) + 2
    psi = torch.from_numpy(inputs.orbitals(96, norb, n).astype(np.float32)).cuda()
    V = torch.from_numpy(inputs.gaussian_potential(96, 0, n).astype(np.float32)).cuda()
    occ = torch.linspace(2.0, 1.0, norb, dtype=torch.float64, device="cuda")

    def run(sel):
        m = len(sel)
        plan = W.Plan([g], [0] * m, prec=W.WVL_F32, graph=False, chain="fused")
        hp = torch.empty((m, g.ncoef), dtype=torch.float32, device="cuda")
        ek = torch.empty(m, dtype=torch.float64, device="cuda")
        ep = torch.empty_like(ek)
        plan.hpsi(psi[sel].reshape(-1), [V], occ[sel], hpsi=hp.view(-1), ekin=ek, epot=ep)
        return hp, ek, ep

    many = run(list(range(norb)))
    assert norb * 2 * n[2] > 2 * 152
    for sel in ([0], [norb - 2, norb - 1]):
        few = run(sel)
        for a, b in zip(many, few):
            assert torch.equal(a[sel], b)
