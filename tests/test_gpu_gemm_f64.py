"""FP64 linear layers at sizes around the tile choice of the FP64 GEMM (rows and outputs that leave
remainders in every tile, counts below one tile and above one tile per SM), through the FP64
forward against the oracle: |d log|psi||, |dE_loc| <= 1e-10 max(1, |x|), the FP64 contract of the
parity tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2307_14123_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14123_gb300 import _build
    _build.build()


@pytest.mark.parametrize("B,width,dets", [(1, 32, 1), (5, 32, 3), (37, 64, 2), (130, 32, 1), (131, 96, 5)])
def test_fp64_forward_over_tile_sizes(B, width, dets):
    from paper_2307_14123_gb300 import Ansatz
    system = fx.molecule("LiH")
    cfg = fx.AnsatzCfg(width, 2, dets)
    th = fx.init_params(system, cfg, 3)
    r = fx.init_walkers(system, B, 5)
    h = Ansatz(system, cfg, "fp64", device="cuda:0")
    la, sg, el = h.local_energy(torch.tensor(th, device="cuda:0"), torch.tensor(r, device="cuda:0"))
    n = min(B, 24)  # the last walkers: the remainders of the tiles
    ref = oracle.Oracle(system, cfg).local_energy(th, r[-n:])
    for got, want in ((la, ref["logabs"]), (el, ref["e_loc"])):
        assert np.all(np.abs(got.cpu().numpy()[-n:] - want) <= 1e-10 * np.maximum(1, np.abs(want)))
    assert np.array_equal(sg.cpu().numpy()[-n:], ref["sign"])
