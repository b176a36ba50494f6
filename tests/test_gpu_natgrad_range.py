"""The natural gradient's passes over the gradients, whose sums are carried in several FP32 terms: they
hold what FP64 sums hold (the accuracy of the centring, sums and solutions past FP32's range or below
it), and the forms that only large calls reach.

Column means: with damping far above the Gram matrix the solution is w / lambda to the last FP32 bit,
so that w = (1, 0, ..), lambda = 1 returns row 0 of the centred gradients.  The sum of 300 values near 1
whose last bits differ is exact in FP64, its mean good to 2^-53; the centred value is rounded to FP32
once (2^-24 of it), and w / (lambda + T) adds less than 2^-30 of it."""
import numpy as np
import pytest
import torch

from paper_2307_14123_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14123_gb300 import _build
    _build.build()


def _handle(name="lih_fp64"):
    from paper_2307_14123_gb300 import Ansatz
    wl = fx.workload(name)
    return Ansatz(wl.system, wl.cfg, "fp32", device=DEV)


def test_centred_gradients_keep_fp64_means():
    h, B = _handle(), 300
    k = np.random.default_rng(3).integers(0, 2, size=(B, h.P))  # steps of 2^-23 above 1
    G = torch.tensor(1.0 + k * 2.0 ** -23, dtype=torch.float32, device=DEV)
    w = torch.zeros(B, device=DEV)
    w[0] = 1.0
    d, _ = h.natural_gradient(G, w, 1.0, max_iter=50, tol=1e-14)
    exact = (k[0] - k.sum(axis=0) / B) * 2.0 ** -23  # integers over 300: to 2^-53 of it
    err = np.abs(d.cpu().numpy().astype(np.float64) - exact)
    assert np.all(err <= (2.0 ** -24 + 2.0 ** -29) * np.abs(exact) + 2.0 ** -52)
