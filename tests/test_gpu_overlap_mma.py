"""The tensor-core scalar products at the edges of their tiles: 128 rows x 64
columns of S, stages of 32 and accumulations of 128 coefficients, slices of whole
accumulations; rows that have no scale (infinity, NaN).

The bound per entry, from the arithmetic: inputs rounded to 2^-56 of their
row's largest magnitude, digit products below 256^-7 of the top ones dropped (6
per coefficient and diagonal), one FP64 addition per slice (at most 304).  With
A = max|a|, B = max|b|, u = 2^-56:
  len A B 8 u + u (A sum|b| + B sum|a|) + 304 2^-53 |a| |b|."""
import numpy as np
import pytest

import oracle.wavelet as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0904_1543_gb300 as W
    return W


def _rows(rng, n, length, dt):
    x = rng.uniform(-1.0, 1.0, (n, length)) * np.exp2(rng.integers(-12, 13, (n, 1)))
    x[:, ::7] *= 2.0 ** -20   # several digits of range inside a row
    return x.astype(dt)


def _check(S, a, b):
    a, b = a.astype(np.float64), b.astype(np.float64)
    rows = sorted({0, a.shape[0] // 2, a.shape[0] - 1})
    cols = sorted({0, b.shape[0] // 2, b.shape[0] - 1})
    ref = O.scalar_products(a[rows], b[cols])
    u = 2.0 ** -56
    A, B = np.abs(a[rows]).max(1), np.abs(b[cols]).max(1)
    bound = (8 * u * a.shape[1] * np.outer(A, B)
             + u * (np.outer(A, np.abs(b[cols]).sum(1)) + np.outer(np.abs(a[rows]).sum(1), B))
             + 304 * 2.0 ** -53 * np.outer(np.linalg.norm(a[rows], axis=1), np.linalg.norm(b[cols], axis=1)))
    assert np.all(np.abs(S[np.ix_(rows, cols)] - ref) <= bound)


@pytest.mark.parametrize("dt", ["float32", "float64"])
@pytest.mark.parametrize("na,nb,length", [
    (1, 1, 1), (2, 3, 31), (5, 64, 32), (127, 65, 33), (128, 63, 127), (129, 64, 128),
    (64, 129, 130), (3, 2, 4099), (9, 5, 60001), (257, 1, 515)])
def test_edges(W, dt, na, nb, length):
    import torch
    rng = np.random.default_rng(na * 1000 + nb + length)
    a, b = _rows(rng, na, length, dt), _rows(rng, nb, length, dt)
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    _check(W.overlap(ta, tb).cpu().numpy(), a, b)
    S = W.overlap(ta).cpu().numpy()
    assert np.array_equal(S, S.T)
    _check(S, a, a)
    assert W.wait_timeouts() == 0


@pytest.mark.parametrize("dt", ["float32", "float64"])
def test_rows_without_a_scale(W, dt):
    """Entries of a row with an infinity or a NaN are what an FP64 sum gives; the others
    are not touched by it; subnormal rows keep their digits."""
    import torch
    rng = np.random.default_rng(5)
    a = _rows(rng, 70, 777, dt)
    a[3, 5], a[66, 700], a[9, 0] = np.inf, -np.inf, np.nan
    a[11] = 0
    a[12] = rng.uniform(0.5, 1.0, 777) * float(np.finfo(dt).tiny) / 8
    S = W.overlap(torch.from_numpy(a).cuda()).cpu().numpy()
    with np.errstate(invalid="ignore", over="ignore"):
        ref = a.astype(np.float64) @ a.astype(np.float64).T
    assert np.array_equal(np.isnan(S), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(S[inf], ref[inf]) and np.array_equal(np.isinf(S), inf)
    keep = [i for i in range(70) if i not in (3, 9, 66)]
    _check(S[np.ix_(keep, keep)], a[keep], a[keep])
    if dt == "float32":
        assert abs(S[12, 12] / ref[12, 12] - 1.0) < 1e-14


@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e25])
@pytest.mark.parametrize("n,length", [(1, 3), (3, 1000), (2, 8193), (700, 40)])
def test_dot_fp32_ranges(W, n, length, scale):
    """FP32 products inside and outside the range of the split sums: FP64
    rounding of a sum of at most 64 terms per thread, 256 threads and 64 blocks."""
    import torch
    rng = np.random.default_rng(length)
    a = (rng.uniform(-1.0, 1.0, (n, length)) * scale).astype("float32")
    b = (rng.uniform(-1.0, 1.0, (n, length)) * scale).astype("float32")
    d = W.dot(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    a, b = a.astype(np.float64), b.astype(np.float64)
    for o in range(0, n, max(1, n // 3)):
        ref = O.scalar_products(a[o:o + 1], b[o:o + 1])[0, 0]
        assert abs(d[o] - ref) <= 384 * 2.0 ** -53 * np.abs(a[o] * b[o]).sum()
