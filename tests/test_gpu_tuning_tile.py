"""The autotuners offer the message register tile only where some launch reads it: not above 16
electrons, whose layers take the sender-tiled and the constant-channel kernels."""
import pytest
import torch

from paper_2307_14123_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14123_gb300 import _build
    _build.build()


def test_message_tile_is_not_timed_where_nothing_reads_it():
    from paper_2307_14123_gb300 import Ansatz, AnsatzBatch
    system, cfg = fx.molecule("C4H4"), fx.AnsatzCfg(32, 2, 1)
    th = torch.tensor(fx.init_params(system, cfg, 1), dtype=torch.float32, device="cuda:0")
    r = torch.tensor(fx.init_walkers(system, 8, 2), dtype=torch.float32, device="cuda:0")
    h = Ansatz(system, cfg, "fp32", device="cuda:0")
    assert h.autotune(th, r)[2] == 8 and h.tile_set()["msg_ib"] == 8
    assert AnsatzBatch([system] * 2, [cfg] * 2, "fp32", device="cuda:0").autotune([th] * 2, [r] * 2)[2] == 8
