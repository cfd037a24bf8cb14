"""Handles of different sizes stepped on two host threads at a time: each thread's results equal those of the
same steps alone. (A kernel's limit of dynamic shared memory is one for all threads.)"""
import threading

import numpy as np
import pytest

from paper_2502_16555_gb300 import workloads as W
from tests._lib import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STEPS = 150


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def march(cfg, kw, ions, out, start=None):
    from paper_2502_16555_gb300 import bte
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            s = bte.Solver(cfg, **kw)
            F = s.initial_state()
            E = torch.from_numpy(W.random_field(cfg["nx"], seed=14, e0=2e3)).cuda()
            ni = torch.full((cfg["nx"],), 1e15, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            if start:
                start.wait(timeout=60)
            for k in range(STEPS):  # a field array: launched kernel by kernel
                if ions:
                    s.ion_step(ni, F, k * cfg["dt_s"])
                else:
                    s.step(F, k * cfg["dt_s"], E=E)
            out.append((F.cpu().numpy(), ni.cpu().numpy()))
    except Exception as e:  # shown by the main thread
        out.append(e)


@pytest.mark.parametrize("kind", ["fp64", "mixed", "structured_fp64", "structured_mixed", "ions"])
def test_two_threads_with_different_grids(kind):
    structured = kind.startswith("structured")
    kw = dict(precision="mixed" if kind.endswith("mixed") else "fp64", structured=structured)
    nx = 100 if kind == "ions" else 6
    cfgs = [W.scaled(W.SMALL, nx=nx, nr=64 if structured else 20 if kind == "ions" else 110, ntheta=9),
            W.scaled(W.SMALL, nx=nx // 2, nr=8, ntheta=3)]
    alone = [[], []]
    for c, o in zip(cfgs, alone):
        march(c, kw, kind == "ions", o)
    both, start = [[], []], threading.Barrier(2)
    ts = [threading.Thread(target=march, args=(c, kw, kind == "ions", o, start)) for c, o in zip(cfgs, both)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for (a,), (b,) in zip(alone, both):
        for r in (a, b):
            if isinstance(r, Exception):
                raise r
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
