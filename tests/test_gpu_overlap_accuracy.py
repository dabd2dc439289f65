"""Scalar products of rows whose large entries do not meet: peaks at different
coefficients, decaying rows, one huge entry beside small ones.  Every entry against the sum of
the magnitudes of its own terms,
  |S_ij - sum_k a_ik b_jk| <= c 2^-53 sum_k |a_ik b_jk|,
with c = 600 from the arithmetic: the digits' error is kept below min(len, 256) 2^-53 of
that sum by the accuracy rule (7 % more for its own rounding) or the entry is an FP64 sum
(chains of at most 320 terms for these lengths), plus one FP64 addition per slice (at most
304)."""
import ctypes

import numpy as np
import pytest

import oracle.wavelet as O


@pytest.fixture(scope="module")
def W():
    import paper_0904_1543_gb300 as W
    return W


@pytest.fixture(scope="module")
def G(W):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return W


def _rows(kind, rng, n, length):
    x = rng.uniform(-1.0, 1.0, (n, length))
    k = np.arange(length)
    if kind == "peaks":        # one huge entry each, at coefficients of its own
        x[np.arange(n), rng.integers(0, length, n)] *= 2.0 ** 60
    elif kind == "gauss":      # localised rows, centres all over, tails below 1e-30
        c, s = rng.uniform(0, length, (n, 1)), length / 24.0
        x = x * np.exp(-(k - c) ** 2 / (2 * s * s)) + 1e-38
    elif kind == "decay":      # from either end, over 28 decades
        d = 10.0 ** (-28.0 * k / length)
        x *= np.where((np.arange(n) % 2 == 0)[:, None], d, d[::-1])
    elif kind == "sparse":     # most entries zero, whole slices of them
        x *= (rng.random((n, length)) < 0.01)
        x[: n // 3, : length // 2] = 0.0
    elif kind == "heavy":      # magnitudes over 16 decades, in any order
        x *= 10.0 ** rng.uniform(-16, 0, (n, length))
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("dt", ["float32", "float64"])
@pytest.mark.parametrize("kind", ["peaks", "gauss", "decay", "sparse", "heavy", "uniform"])
@pytest.mark.parametrize("na,nb,length", [(5, 7, 40), (33, 20, 515), (70, 130, 3001), (140, 40, 20004)])
def test_relative_to_own_terms(G, dt, kind, na, nb, length):
    import torch
    rng = np.random.default_rng(na + length)
    a = _rows(kind, rng, na, length).astype(dt)
    b = _rows(kind, rng, nb, length).astype(dt)
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    S, Q = G.overlap(ta, tb).cpu().numpy(), G.overlap(ta).cpu().numpy()
    assert np.array_equal(Q, Q.T)
    a, b = a.astype(np.float64), b.astype(np.float64)
    rows, cols = sorted({0, 1, na // 2, na - 1}), sorted({0, 3, nb // 2, nb - 1})
    for got, y, js in ((S, b, cols), (Q, a, rows)):
        ref = O.scalar_products(a[rows], y[js])
        own = np.abs(a[rows]) @ np.abs(y[js]).T
        err = np.abs(got[np.ix_(rows, js)] - ref)
        assert np.all(err <= 600 * 2.0 ** -53 * own), float((err / np.maximum(own, 1e-300)).max() * 2.0 ** 53)
    assert G.wait_timeouts() == 0


@pytest.mark.gpu
def test_lost_terms(G):
    """The smallest examples: terms that meet only where neither row is large."""
    import torch
    for dt in (torch.float32, torch.float64):
        for length in (2, 1024):
            a = torch.zeros((1, length), dtype=dt, device="cuda")
            b = torch.zeros((1, length), dtype=dt, device="cuda")
            a[0, 0], a[0, 1], b[0, 1] = 2.0 ** 60, 1.0, 1.0
            assert float(G.overlap(a, b)) == 1.0
            a[0, 0], a[0, 1], b[0, 0], b[0, 1] = 1.0, 1e-10, 1e-10, 1.0
            ref = float(a[0, 0].double() * b[0, 0].double() + a[0, 1].double() * b[0, 1].double())
            assert abs(float(G.overlap(a, b)) / ref - 1.0) < 4e-16


def _size(W, na, nb, length, prec):
    need = ctypes.c_size_t(0)
    assert W.lib().wvl_overlap_workspace_size(prec, na, nb, length, ctypes.byref(need)) == 0
    return need.value


def test_workspace_grows_with_every_size(W):
    """A workspace for the largest block serves every smaller one; and its size is of the order of
    the result's, not of the number of slices times it."""
    for length in (1, 300, 20000, 884736, 40000000):
        last = 0
        for n in (1, 2, 31, 64, 200, 255, 256, 257, 300, 700, 1000, 1023, 1024, 1156, 2048, 4099, 8192):
            s = _size(W, n, n, length, W.WVL_F32)
            assert s >= last and s >= _size(W, n, 1, length, W.WVL_F32)
            assert s >= _size(W, n, n, max(1, length // 3), W.WVL_F32)
            last = s
            if length <= 884736:
                assert s <= 20 * n * n + (64 << 20), (n, s)


@pytest.mark.gpu
def test_workspace_of_the_largest_block(G):
    import torch
    lib, length = G.lib(), 5000
    x = torch.rand((400, length), device="cuda") - 0.5
    need = _size(G, 400, 400, length, G.WVL_F32)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    for n in (1, 3, 40, 129, 250, 311, 399, 400):
        for m in (1, n):
            S = torch.full((n, m), 7.0, dtype=torch.float64, device="cuda")
            r = lib.wvl_overlap(G.WVL_F32, n, x.data_ptr(), m, x[1:].data_ptr() if n < 400 else x.data_ptr(),
                                length, S.data_ptr(), ws.data_ptr(), need, None)
            assert r == 0, (n, m)
            y = (x[1:] if n < 400 else x)[:m]
            torch.cuda.synchronize()
            assert torch.allclose(S, x[:n].double() @ y.double().T, rtol=0, atol=1e-9)
