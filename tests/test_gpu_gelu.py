"""Both device forms of the network's activation, GELU(z) = z Phi(z) with erf by
Abramowitz & Stegun 7.1.26: the inference form (approximate reciprocal with a
Newton step, hardware exponential, |z| clamped) and the training form (rounded
reciprocal, library exponential), against the exact erf and at special values.
The bound is the one test_gelu_bound.py states for the formula in FP32, which
describes the training form's arithmetic: 4e-7 (1 + |z|)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gelu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_03067_gb300 import build, mpm
    build.build()
    return lambda z: [t.cpu().numpy() for t in mpm.mpm_debug_gelu(torch.from_numpy(z).cuda())]


def exact(z):
    return np.array([0.5 * v * math.erfc(-v / math.sqrt(2.0)) for v in z.astype(np.float64)])


def test_error_against_the_exact_erf(gelu):
    z = np.concatenate([np.linspace(-10.0, 10.0, 400001), np.linspace(-1e-2, 1e-2, 20001),
                        -np.logspace(-38, 38, 5000), np.logspace(-38, 38, 5000)]).astype(np.float32)
    want = exact(z)
    inference, train = (g.astype(np.float64) for g in gelu(z))
    for got in (inference, train):
        assert np.all(np.abs(got - want) <= 4e-7 * (1.0 + np.abs(z.astype(np.float64))))
    # no further off than the training form, but for the last bit of a result below |z|
    worst, worst_train = (np.max(np.abs(g - want) / (1e-30 + np.abs(z.astype(np.float64)))) for g in (inference, train))
    print(f"max error / |z|: inference {worst:.3e}, training {worst_train:.3e}")
    assert worst <= worst_train + 2.0 ** -24


def test_special_values(gelu):
    big = np.float32(3.4e38)
    z = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, big, -big, 1e4, -1e4, 2e4, -2e4, 1e-40, -1e-40, 30.0, -30.0],
                 np.float32)
    for g in gelu(z):
        assert g[0] == 0.0 and g[1] == 0.0
        assert g[2] == np.inf and np.isnan(g[3]) and np.isnan(g[4])
        assert np.array_equal(g[[5, 7, 9, 13]], z[[5, 7, 9, 13]])
        assert np.all(g[[6, 8, 10]] == 0.0) and abs(g[14]) < 1e-30
        assert abs(g[11] - 5e-41) < 1e-44 and abs(g[12] + 5e-41) < 1e-44
