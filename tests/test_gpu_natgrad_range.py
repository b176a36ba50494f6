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


def _tiles(n, tri):
    """Output tiles of an n x n Gram matrix: 256 x 128, all or those that reach row >= column."""
    mp, nt = -(-n // 256), -(-n // 128)
    return mp * (mp - 1) + min(2 * mp, nt) if tri else mp * nt


def _waves(n, chunks, tri):
    """Fewest waves of tiles over the chunks per launch (1 to 16), and that number of chunks."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return min((chunks // j * -(-j * _tiles(n, tri) // sms) + -(-(chunks % j) * _tiles(n, tri) // sms), -j)
               for j in range(1, 17))


def _solve64(G, w, lam):
    Gc = G.double() - G.double().mean(dim=0)
    T = Gc @ Gc.t() / G.shape[0]
    T.diagonal().add_(lam)
    return torch.linalg.solve(T, w.double()) @ Gc


def _synthetic(B, P, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    G = torch.randn(B, P, device=DEV, generator=g) * (0.05 + 1.95 * torch.rand(P, device=DEV, generator=g))
    G += torch.randn(P, device=DEV, generator=g)
    w = torch.randn(B, device=DEV, generator=g)
    return G, (2.0 / B) * (w - w.mean())


def test_triangular_gram_over_several_launches():
    """600 walkers x 400,000 parameters: the half of the Gram matrix that is computed saves waves, its
    chunks take several launches, and the last row and column blocks are ragged.  Against a dense FP64
    solution, with the bound of the other parity tests (condition below 1e3)."""
    h, B = _handle("n2_fp32"), 600
    chunks = -(-h.P // 8192)
    (full, _), (half, j) = _waves(B, chunks, False), _waves(B, chunks, True)
    assert half < full and chunks > 2 * -j
    G, w = _synthetic(B, h.P, 1)
    lam = 0.1 * float(G.double().var(dim=0, unbiased=False).sum()) / B
    d, st = h.natural_gradient(G, w, lam, max_iter=400, tol=1e-9)
    ref = _solve64(G, w, lam)
    assert float(st[1]) <= 1e-9 and float((d.double() - ref).norm()) <= 2e-3 * float(ref.norm())


@pytest.mark.parametrize("B", [9514, 9515])
def test_largest_one_kernel_solve_and_the_loop(B):
    """The largest system of the one-kernel solve and the smallest of the launches per iteration,
    against a dense FP64 solution (condition below 1e3: the largest eigenvalue of the random matrix is
    about four times the mean)."""
    from paper_2307_14123_gb300 import Ansatz
    h = Ansatz(fx.molecule("H"), fx.AnsatzCfg(32, 1, 1), "fp32", device=DEV)
    G, w = _synthetic(B, h.P, 2)
    d, st = h.natural_gradient(G, w, -0.1, max_iter=400, tol=1e-9)
    ref = _solve64(G, w, float(st[3]))
    assert 1 <= float(st[0]) < 400 and float(st[1]) <= 1e-9
    assert float((d.double() - ref).norm()) <= 2e-3 * float(ref.norm())
