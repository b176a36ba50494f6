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


def test_column_sums_past_fp32():
    """A parameter whose gradient is 3e37 for all 300 walkers has a sum of 9e39, a mean of 3e37 and a
    centred gradient of zero, as if it were zero."""
    h, B = _handle(), 300
    rng = np.random.default_rng(4)
    G = torch.tensor(rng.standard_normal((B, h.P)), dtype=torch.float32, device=DEV)
    w = torch.tensor(rng.standard_normal(B) / B, dtype=torch.float32, device=DEV)
    G[:, 7] = 0.0
    ref, _ = h.natural_gradient(G, w, -0.1, max_iter=200, tol=1e-9)
    G[:, 7] = 3e37
    d, _ = h.natural_gradient(G, w, -0.1, max_iter=200, tol=1e-9)
    assert bool(torch.isfinite(ref).all()) and torch.equal(d, ref)


@pytest.mark.parametrize("g_exp,w_exp", [(-20, 100), (0, 100), (20, -100), (0, -100)])
def test_solutions_outside_fp32(g_exp, w_exp):
    """Powers of two pass through the call exactly: gradients times 2^g, weights times 2^w give the
    direction times 2^(w - g), bit for bit, also where the solution (of order 2^(w - 2 g)) is past
    FP32's range or below it."""
    h, B = _handle(), 200
    rng = np.random.default_rng(5)
    G = torch.tensor(rng.standard_normal((B, h.P)), dtype=torch.float32, device=DEV)
    w = torch.tensor(rng.standard_normal(B), dtype=torch.float32, device=DEV)
    ref, st = h.natural_gradient(G, w, -0.1, max_iter=200, tol=1e-9)
    d, st2 = h.natural_gradient(G * 2.0 ** g_exp, w * 2.0 ** w_exp, -0.1, max_iter=200, tol=1e-9)
    assert float(st[0]) == float(st2[0])
    want = ref.double() * 2.0 ** (w_exp - g_exp)
    normal = want.abs() >= 2.0 ** -126  # (below, FP32 results have fewer bits)
    assert float(normal.double().mean()) > 0.5
    assert torch.equal(d.double()[normal], want[normal])
