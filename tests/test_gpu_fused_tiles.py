"""The fused layer kernel over the ways its tiles of whole electrons are cut: one tile per walker (4
electrons), a last tile without electrons (12: the Laplacian and the value channel alone), unequal
spin blocks (8 + 4, 5 + 2, 8 + 1), with constant and with node-mapped channels.  Against the oracle
under the FP32 contract, and the separate layer kernels within its bounds."""
import os

import numpy as np
import pytest
import torch

import oracle
from fp32_contract import check_fp32_oracle, near_nodal
from paper_2307_14123_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14123_gb300 import _build
    _build.build()
    oracle.build()
    oracle.Oracle.set_threads(os.cpu_count() or 1)


@pytest.mark.parametrize("n_up,n_dn,Z", [(2, 2, (3, 1)), (6, 6, (6, 6)), (8, 4, (8, 4)), (5, 2, (5, 2)),
                                         (8, 1, (5, 4))])
def test_tile_cuts(n_up, n_dn, Z):
    from paper_2307_14123_gb300 import Ansatz
    system = fx.System(Z=np.array(Z, float), R=np.array([[0, 0, 1.1], [0.3, 0, -1.2]]), n_up=n_up, n_down=n_dn)
    cfg = fx.AnsatzCfg(128, 2, 2)
    th = fx.init_params(system, cfg, 8).astype(np.float32).astype(np.float64)
    r = fx.init_walkers(system, 8, 6).astype(np.float32).astype(np.float64)
    h = Ansatz(system, cfg, "fp32", device=DEV)
    o = oracle.Oracle(system, cfg)
    ref = o.local_energy(th, r, with_grad=True)
    out = {}
    for mode in (1, 2):
        h.set_layer_kernel(mode)
        assert h.layer_kernel_fused() == (mode == 1)
        out[mode] = [v.cpu().numpy().astype(np.float64) for v in h.local_energy(
            torch.tensor(th, dtype=torch.float32, device=DEV), torch.tensor(r, dtype=torch.float32, device=DEV))]
        assert h.device_status() & 0x4 == 0
        check_fp32_oracle(f"{n_up} + {n_dn}, layer kernel {mode}", *out[mode], o, th, r, ref=ref, max_exception_frac=0.34)
    ok = ~near_nodal(o, th, r, ref["logabs"])
    S = 0.5 * (np.abs(ref["lap"]) + np.sum(ref["grad"] ** 2, axis=1))
    assert ok.any()
    assert np.all(np.abs(out[1][0] - out[2][0])[ok] <= 1e-5 * np.maximum(1, np.abs(ref["logabs"][ok])))
    assert np.all(np.abs(out[1][2] - out[2][2])[ok] <= np.maximum(1e-4, 1e-5 * S[ok]))
