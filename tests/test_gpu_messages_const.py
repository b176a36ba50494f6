"""The message kernel of constant node channels (layer 0 on spin embeddings) against the general kernel,
which message-kernel mode 1 takes in every layer: the same sums in the same order with the same
roundings, so the same bits, in FP32 and as BF16 operands, at the widths of its four, two and one
features per lane, below and above the split of the messages (nine electrons), and for an empty spin
block.  Above 16 electrons one layer only: the later ones take the sender-tiled kernel by default."""
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


@pytest.mark.parametrize("mol,width,layers,B", [("LiH", 64, 2, 33), ("H2O", 96, 2, 9), ("NH3", 128, 2, 9), ("H", 32, 2, 5),
                                                ("N2", 192, 2, 6), ("C4H4", 256, 1, 4), ("C6H6", 32, 1, 3),
                                                ("7 up", 64, 2, 6)])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_constant_channels_have_the_general_bits(mol, width, layers, B, precision):
    from paper_2307_14123_gb300 import Ansatz
    if precision == "bf16" and width % 64:
        pytest.skip("BF16 mode takes widths in multiples of 64")
    system = (fx.System(Z=np.array([5.0, 2.0]), R=np.array([[0, 0, 1.1], [0.3, 0, -1.2]]), n_up=7, n_down=0)
              if mol == "7 up" else fx.molecule(mol))
    cfg = fx.AnsatzCfg(width, layers, 2)
    h = Ansatz(system, cfg, precision, device=DEV)
    th = torch.tensor(fx.init_params(system, cfg, 11), dtype=torch.float32, device=DEV)
    r = torch.tensor(fx.init_walkers(system, B, 12), dtype=torch.float32, device=DEV)
    h.set_layer_kernel(2)
    a = h.local_energy(th, r)
    h.set_msg_kernel(1)
    b = h.local_energy(th, r)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
