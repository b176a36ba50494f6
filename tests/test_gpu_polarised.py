"""Fully polarised systems past the fused kernel's size (no spin-down electrons: one spin block is
empty) in the FP32 modes, whose jet messages take the sender-tiled kernel: with its w' and w''
tables in shared memory (18 electrons) and read from global memory (24, the largest block).

FP32 under the FP32 contract against the oracle; the sender-tiled and the general kernel (the same
messages, summed in different orders) against each other, FP32 within the contract's bounds and
BF16 within the BF16 mode's (a message may round to the other BF16 neighbour), outside the
contract's exception class."""
import itertools
import os

import numpy as np
import pytest
import torch

import oracle
from fp32_contract import bf16_logabs_bound, check_fp32_oracle, near_nodal
from paper_2307_14123_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14123_gb300 import _build
    _build.build()
    oracle.build()
    oracle.Oracle.set_threads(os.cpu_count() or 1)


def _case(n_up, B=5, K=2):
    """n_up hydrogen nuclei on a grid, the envelope of every orbital largest at its own nucleus, so
    that the one large matrix per determinant is well conditioned."""
    R = 4.0 * np.array(list(itertools.product(range(3), repeat=3))[:n_up])
    system, cfg = fx.System(Z=np.ones(n_up), R=R, n_up=n_up, n_down=0), fx.AnsatzCfg(64, 2, K)
    th = fx.init_params(system, cfg, 5)
    off = fx.param_offsets(system, cfg)
    o = off["omega_up"][0]
    th[o:o + K * n_up * n_up] = np.tile(0.05 + np.eye(n_up), (K, 1)).ravel()
    o = off["b_o_up"][0]
    th[o:o + K * n_up] = 3.0
    th = th.astype(np.float32).astype(np.float64)
    r = fx.init_walkers(system, B, 6).astype(np.float32).astype(np.float64)
    return system, cfg, th, r


@pytest.mark.parametrize("n_up", [18, 24])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_empty_spin_block(n_up, precision):
    from paper_2307_14123_gb300 import Ansatz
    system, cfg, th, r = _case(n_up)
    h = Ansatz(system, cfg, precision, device="cuda:0")
    assert h.msg_kernel() == 2
    tht = torch.tensor(th, dtype=torch.float32, device="cuda:0")
    rt = torch.tensor(r, dtype=torch.float32, device="cuda:0")
    out = {}
    for mode in (2, 1):
        h.set_msg_kernel(mode)
        out[mode] = [v.cpu().numpy().astype(np.float64) for v in h.local_energy(tht, rt)]
        assert h.device_status() & 0x4 == 0
    o = oracle.Oracle(system, cfg)
    ref = o.local_energy(th, r, with_grad=True)
    S = 0.5 * (np.abs(ref["lap"]) + np.sum(ref["grad"] ** 2, axis=1))
    ok = ~near_nodal(o, th, r, ref["logabs"])
    (la2, sg2, el2), (la1, sg1, el1) = out[2], out[1]
    print(f"{n_up} {precision}: {ok.sum()} walkers outside the exception class, tiled vs general max |d log|psi|| "
          f"{np.max(np.abs(la2 - la1)):.2e}, max |dE|/S {np.max(np.abs(el2 - el1) / S):.2e}")
    if precision == "fp32":
        for mode in (2, 1):
            check_fp32_oracle(f"{n_up} up, kernel {mode}", *out[mode], o, th, r, ref=ref, max_exception_frac=0.34)
        la_tol, e_tol = 1e-5 * np.maximum(1, np.abs(ref["logabs"])), np.maximum(1e-4, 1e-5 * S)
    else:
        la_tol, e_tol = bf16_logabs_bound(o, th, r, ref["logabs"]), np.maximum(1e-2, 2e-2 * S)
    assert ok.any()
    assert np.all(np.isfinite(el2)) and np.all(np.isfinite(la2))
    assert np.all(np.abs(la2 - la1)[ok] <= la_tol[ok])
    assert np.all(np.abs(el2 - el1)[ok] <= e_tol[ok])
    assert np.array_equal(sg2[ok], sg1[ok])
