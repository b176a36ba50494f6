"""Two host threads with handles of different sizes, each on a stream of its own: the calls of one
must not change what the other's launches are allowed (the shared-memory limit belongs to a kernel,
not to a launch), and each gives the results that it gives alone, bit for bit.  C2H4 (216 edges)
needs more than the default 48 KB of a block in the message kernels of the value forward and of the
reverse pass, LiH (14 edges) does not."""
import threading

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


def test_two_threads_of_different_sizes():
    from paper_2307_14123_gb300 import Ansatz
    jobs = []
    for mol in ("C2H4", "LiH"):
        system, cfg = fx.molecule(mol), fx.AnsatzCfg(32, 2, 1)
        h = Ansatz(system, cfg, "fp64", device=DEV)
        th = torch.tensor(fx.init_params(system, cfg, 3), device=DEV)
        r = torch.tensor(fx.init_walkers(system, 4, 4), device=DEV)
        w = torch.tensor(np.linspace(-1, 1, 4), device=DEV)
        jobs.append((h, th, r, w, torch.cuda.Stream()))

    def once(h, th, r, w):
        return [*h.ansatz_eval(th, r), h.grad_logpsi(th, r, w, 0)]

    alone = [once(*j[:4]) for j in jobs]
    torch.cuda.synchronize()
    faults, start = [], threading.Barrier(2)

    def work(k):
        h, th, r, w, stream = jobs[k]
        try:
            with torch.cuda.stream(stream):
                start.wait()
                for _ in range(300):
                    out = once(h, th, r, w)
                stream.synchronize()
            assert all(torch.equal(x, y) for x, y in zip(out, alone[k]))
        except BaseException as e:  # noqa: BLE001 (handed to the test's thread)
            faults.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults
