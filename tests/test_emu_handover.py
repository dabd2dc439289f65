"""Accuracy of the tensor-core passes on fields whose lines differ by many orders of
magnitude: the error of every element against the stated bound of a convolution, 2^-52 max|f|
max|x| over its own line, carried through the three passes; the lines of passes 2 and 3 have
scales of their own although the passes hand integers over.  And the arithmetic of the
hand-over on the CPU (tests/emu_handover_check.cpp includes the library's own header)."""
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import oracle.filters as F
import oracle.wavelet as O
from paper_0904_1543_gb300 import inputs

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_handover_arithmetic():
    cxx = shutil.which("g++")
    inc = next((os.path.join(d, "include") for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda")
                if d and os.path.exists(os.path.join(d, "include", "cuda_runtime_api.h"))), None)
    if cxx is None or inc is None:
        pytest.skip("needs g++ and the CUDA headers")
    with tempfile.TemporaryDirectory() as td:
        exe = os.path.join(td, "check")
        r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_0904_1543_gb300", "csrc"),
                            "-I", os.path.join(ROOT, "include"), "-I", inc,
                            os.path.join(HERE, "emu_handover_check.cpp"), "-o", exe],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0 and "OK" in r.stdout, r.stdout[-3000:]


def _fields(n, shape):
    """A Gaussian of 2.5 points (its tails fall below 1e-30 of its peak), and fields of 1e-9
    with one line of large values along each axis."""
    N3, N2, N1 = shape
    z, y, x = np.meshgrid(np.arange(N3), np.arange(N2), np.arange(N1), indexing="ij")
    r2 = (x - N1 // 2) ** 2 + (y - N2 // 2) ** 2 + (z - N3 // 2) ** 2
    out = [np.exp(-r2 / (2 * 2.5 ** 2))]
    for axis in range(3):
        f = 1e-9 * inputs.random_field(471, axis, (1,) + shape)[0]
        at = [1, 2, 1]
        at[2 - axis] = slice(None)
        f[tuple(at)] += inputs.random_field(472, axis, (1, N3 + N2 + N1))[0][:shape[2 - axis]]
        out.append(f)
    return np.stack(out)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(12, 16, 20), (9, 17, 5), (24, 24, 24), (3, 40, 2)])
@pytest.mark.parametrize("transposed", [False, True])
def test_error_over_own_line(n, transposed):
    import torch
    import paper_0904_1543_gb300 as W
    g = W.Grid(n)
    x = _fields(n, g.fine)
    got = (W.magicfilter_T if transposed else W.magicfilter)(torch.from_numpy(x).cuda(), g, emu=True)
    got = got.cpu().numpy().astype(np.longdouble)
    w, k0 = F.magic()
    w = np.abs(np.asarray(w))
    sgn = -1 if transposed else 1
    for k in range(len(x)):
        u, err = x[k].astype(np.longdouble), np.zeros(g.fine)
        for axis in (2, 1, 0):   # along x, then y, then z
            lmax = np.max(np.abs(u) + err, axis=axis, keepdims=True).astype(np.float64)
            err = sum(w[t] * np.roll(err, sgn * (k0 + t), axis) for t in range(F.NTAP))
            err = err + 2.0 ** -52 * w.max() * lmax
            u = (O.magicfilter_T_1d if transposed else O.magicfilter_1d)(u, axis)
        # and one rounding to FP64
        bad = np.abs(got[k] - u) > err + 2.0 ** -53 * np.abs(u).astype(np.float64)
        assert not bad.any(), (k, int(bad.sum()), float((np.abs(got[k] - u) / err).max()))
    assert W.wait_timeouts() == 0
