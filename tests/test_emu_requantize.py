"""CPU check of the integers that the tensor-core passes hand over (the C++ program
tests/emu_requantize_check.cpp includes the library's own header), and the
GPU form at cells where tiles, windows and line groups are cut short."""
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import oracle.wavelet as O
from paper_0904_1543_gb300 import inputs

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_requantize():
    cxx = shutil.which("g++")
    inc = next((os.path.join(d, "include") for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda")
                if d and os.path.exists(os.path.join(d, "include", "cuda_runtime_api.h"))), None)
    if cxx is None or inc is None:
        pytest.skip("needs g++ and the CUDA headers")
    with tempfile.TemporaryDirectory() as td:
        exe = os.path.join(td, "check")
        r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_0904_1543_gb300", "csrc"),
                            "-I", os.path.join(ROOT, "include"), "-I", inc,
                            os.path.join(HERE, "emu_requantize_check.cpp"), "-o", exe],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0 and "OK" in r.stdout, r.stdout[-3000:]


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(1, 1, 1), (1, 5, 2), (7, 1, 4), (8, 8, 8), (9, 4, 17), (33, 3, 2)])
def test_chain_on_cut_tiles(n):
    """Lines shorter than a window, extents that are no multiple of 16, fewer lines than a
    tile, orbitals of very different magnitude: 1e-12 of each orbital's own largest value, the
    form's stated accuracy."""
    import torch
    import paper_0904_1543_gb300 as W
    g = W.Grid(n, (0.25, 0.3, 0.2))
    psi = inputs.orbitals(91, 3, n) * np.array([1.0, 1e-30, 1e12])[:, None]
    V = inputs.gaussian_potential(91, 0, n)
    occ = np.array([2.0, 1.0, 0.5])
    hp, ek, ep = W.hpsi_local(torch.from_numpy(psi).cuda(), torch.from_numpy(V).cuda(),
                              torch.from_numpy(occ).cuda(), g, emu=True)
    s = W.synthesis(torch.from_numpy(psi).cuda(), g, emu=True).cpu().numpy()
    for o in range(3):
        r = O.hpsi_local(psi[o], V, occ[o], n, (0.25, 0.3, 0.2))
        assert np.abs(hp[o].cpu().numpy() - r["hpsi_c"]).max() <= 1e-12 * np.abs(r["hpsi_c"]).max()
        ref = O.synthesis3d(O.uncompress(psi[o], n))
        assert np.abs(s[o] - ref).max() <= 1e-12 * np.abs(ref).max()
    assert W.wait_timeouts() == 0
