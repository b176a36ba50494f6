"""The separate layer kernels over the sizes where their splits and vectors change: widths that are
not a multiple of the wide vectors, electron counts on both sides of the split messages (nine) and
edge counts on both sides of the staged filter slices, few and many walkers (16 and 32 edges per
block of the hidden layer).  Against the oracle: FP64 to the parity tests' 1e-10, for E_loc relative
to the size S_b of the kinetic terms whose difference it is (gradient directions 1e-8 of their
largest), FP32 under the FP32 contract."""
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


def _inputs(mol, width, layers, dets, B, dtype):
    system, cfg = fx.molecule(mol), fx.AnsatzCfg(width, layers, dets)
    th = fx.init_params(system, cfg, 11).astype(dtype).astype(np.float64)
    r = fx.init_walkers(system, B, 12).astype(dtype).astype(np.float64)
    return system, cfg, th, r


@pytest.mark.parametrize("mol,width,B", [("LiH", 160, 3), ("H2O", 96, 3), ("N2", 32, 2), ("C4H4", 32, 1),
                                         ("LiH", 32, 1500), ("H", 32, 7)])
def test_fp64_energies_and_gradients(mol, width, B):
    from paper_2307_14123_gb300 import Ansatz
    system, cfg, th, r = _inputs(mol, width, 2, 2, B, np.float64)
    h = Ansatz(system, cfg, "fp64", device=DEV)
    tht, rt = torch.tensor(th, device=DEV), torch.tensor(r, device=DEV)
    la, sg, el = h.local_energy(tht, rt)
    n = min(B, 6)  # the last walkers
    o = oracle.Oracle(system, cfg)
    ref = o.local_energy(th, r[-n:], with_grad=True)
    S = 0.5 * (np.abs(ref["lap"]) + np.sum(ref["grad"] ** 2, axis=1))
    for got, want, size in ((la, ref["logabs"], np.abs(ref["logabs"])), (el, ref["e_loc"], S)):
        assert np.all(np.abs(got.cpu().numpy()[-n:] - want) <= 1e-10 * np.maximum(1, size))
    assert np.array_equal(sg.cpu().numpy()[-n:], ref["sign"])
    w = np.random.default_rng(1).normal(size=n)
    g = h.grad_logpsi(tht, rt[-n:].contiguous(), torch.tensor(w, device=DEV), 0).cpu().numpy()
    dirs = np.random.default_rng(2).normal(size=(3, o.P))
    want = w @ o.grad_jvp(th, r[-n:], dirs)
    assert np.all(np.abs(dirs @ g - want) <= 1e-8 * max(1, np.abs(want).max()))


@pytest.mark.parametrize("mol,width,B", [("LiH", 32, 12), ("LiH", 64, 12), ("H2O", 96, 8), ("NH3", 128, 8), ("N2", 64, 6),
                                         ("C4H4", 64, 3), ("C6H6", 32, 2)])
def test_fp32_separate_layers(mol, width, B):
    """Constant node channels in the first layer and node-mapped ones in the second."""
    from paper_2307_14123_gb300 import Ansatz
    system, cfg, th, r = _inputs(mol, width, 2, 2, B, np.float32)
    h = Ansatz(system, cfg, "fp32", device=DEV)
    h.set_layer_kernel(2)
    la, sg, el = h.local_energy(torch.tensor(th, dtype=torch.float32, device=DEV),
                                torch.tensor(r, dtype=torch.float32, device=DEV))
    assert h.device_status() == 0
    check_fp32_oracle(f"{mol} D={width}", la.cpu().numpy(), sg.cpu().numpy(), el.cpu().numpy(),
                      oracle.Oracle(system, cfg), th, r, max_exception_frac=0.34)
