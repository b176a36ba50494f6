"""Distance features (n_rbf) and widths at which the edge hidden layer's weights nearly fill a block's
shared memory, with rows for its smaller blocks (40 LiH walkers, 560 edges) and for its larger ones
(1500, 21,000 edges): a walker's results do not depend on the walkers beside it, so the 40 walkers
alone give the bits that they give among the 1500.  Against the oracle, the last walkers: FP64 to
1e-10 (E_loc relative to the size S_b of its kinetic terms), FP32 at the widths of the FP32 contract."""
import numpy as np
import pytest
import torch

import oracle
from fp32_contract import check_fp32_oracle
from paper_2307_14123_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14123_gb300 import _build
    _build.build()


# values_only: the jets' features and the weights together pass a block's shared memory
@pytest.mark.parametrize("precision,n_rbf,width,values_only", [
    ("fp64", 16, 512, 0), ("fp64", 32, 256, 0), ("fp64", 64, 96, 0), ("fp64", 40, 224, 1), ("fp64", 8, 32, 0),
    ("fp32", 64, 256, 0), ("fp32", 40, 416, 0), ("fp32", 48, 384, 1), ("fp32", 56, 320, 1), ("fp32", 16, 512, 0)])
def test_hidden_layer_shapes(precision, n_rbf, width, values_only):
    from paper_2307_14123_gb300 import Ansatz
    system, cfg = fx.molecule("LiH"), fx.AnsatzCfg(width, 2, 2, n_rbf)
    dtype = np.float64 if precision == "fp64" else np.float32
    th = fx.init_params(system, cfg, 11).astype(dtype).astype(np.float64)
    r = fx.init_walkers(system, 1500, 12).astype(dtype).astype(np.float64)
    h = Ansatz(system, cfg, precision, device=DEV)
    tht, rt = (torch.tensor(v.astype(dtype), device=DEV) for v in (th, r))
    few = rt[-40:].contiguous()
    for f in (h.ansatz_eval,) if values_only else (h.ansatz_eval, h.local_energy):
        many = f(tht, rt)
        for x, y in zip(many, f(tht, few)):
            assert bool(torch.isfinite(x).all()) and torch.equal(x[-40:], y)
    assert h.device_status() == 0
    if values_only or (precision == "fp32" and width > 256):
        return
    n = 4
    la, sg, el = (v.cpu().numpy()[-n:].astype(np.float64) for v in many)
    o = oracle.Oracle(system, cfg)
    ref = o.local_energy(th, r[-n:], with_grad=True)
    if precision == "fp32":
        check_fp32_oracle(f"n_rbf={n_rbf} D={width}", la, sg, el, o, th, r[-n:], ref=ref, max_exception_frac=0.34)
    else:
        S = 0.5 * (np.abs(ref["lap"]) + np.sum(ref["grad"] ** 2, axis=1))
        assert np.array_equal(sg, ref["sign"])
        assert np.all(np.abs(la - ref["logabs"]) <= 1e-10 * np.maximum(1, np.abs(ref["logabs"])))
        assert np.all(np.abs(el - ref["e_loc"]) <= 1e-10 * np.maximum(1, S))
