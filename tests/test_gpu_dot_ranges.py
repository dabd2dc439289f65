"""FP32 scalar products whose terms leave the range of the split sums, all or in part: zeros,
magnitudes far below and above one, infinities and NaN.  The bound of the sums: FP64 rounding
of at most 64 terms per thread, 256 threads and 64 blocks."""
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


@pytest.mark.parametrize("length", [1, 7, 1000, 4099, 70000])
def test_ranges(W, length):
    import torch
    rng = np.random.default_rng(length)
    scale = [0.0, 1e-9, 1e-12, 1e-15, 1e-22, 1e-30, 1e-42, 1e12, 1e18, 1e30]
    a = rng.uniform(-1.0, 1.0, (2 * len(scale), length))
    b = rng.uniform(-1.0, 1.0, (2 * len(scale), length))
    for i, s in enumerate(scale):
        a[i] *= s
        b[i] *= s
        a[len(scale) + i] *= s                    # one side only
        b[len(scale) + i, ::2] = 0.0              # and half of the other zero
    a, b = a.astype("float32"), b.astype("float32")
    d = W.dot(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    a, b = a.astype(np.float64), b.astype(np.float64)
    for o in range(a.shape[0]):
        ref = O.scalar_products(a[o:o + 1], b[o:o + 1])[0, 0]
        assert abs(d[o] - ref) <= 384 * 2.0 ** -53 * np.abs(a[o] * b[o]).sum(), o


def test_not_finite(W):
    import torch
    a = np.zeros((6, 515), dtype="float32")
    b = np.zeros((6, 515), dtype="float32")
    a[0, 3] = np.inf               # inf * 0
    a[1, 3], b[1, 3] = np.inf, 2.0
    a[2, 514] = np.nan
    a[3, 0], b[3, 0], a[3, 1], b[3, 1] = 3e38, 3e38, 3e38, -3e38   # products beyond FP32
    a[4, :], b[4, :] = 1e-40, 1e-40                                # subnormal factors
    a[5, 0], b[5, 0], a[5, 9], b[5, 9] = 3e38, 2.0, 1e-40, 1e-40
    d = W.dot(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.isnan(d[0]) and d[1] == np.inf and np.isnan(d[2]) and d[3] == 0.0
    f = np.float64
    assert abs(d[4] / (515 * f(a[4, 0]) ** 2) - 1) < 1e-13
    assert abs(d[5] / (f(a[5, 0]) * 2.0) - 1) < 1e-15
