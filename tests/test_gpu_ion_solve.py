"""The ion system's elimination (csrc/bte_hybrid.cu) at the edges of its chunks of 32 columns, right-hand side
included, in the shared-memory branch. The density after one ion step against the oracle; tolerance that of
the parity tests, 1e-10."""
import numpy as np
import pytest

from oracle import bte as O
from oracle import hybrid as H
from paper_2502_16555_gb300 import workloads as W
from tests._lib import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("nx", [3, 31, 32, 33, 63, 64, 65, 127, 128, 129])
def test_ion_solve_chunk_edges(nx):
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=nx, nr=6, ntheta=4)
    ops = O.Operators(cfg)
    F = ops.initial_state()
    x = np.linspace(-1.0, 1.0, nx)
    ni = 1e15 * (1.05 - 0.9 * x * x)
    t = 0.13 / cfg["freq_Hz"]
    ref = H.Hybrid(ops).ion_step(ni, F, t)
    n = torch.from_numpy(ni.copy()).cuda()
    bte.Solver(cfg, precision="fp64").ion_step(n, torch.from_numpy(F).cuda(), t)
    err = float(np.linalg.norm(n.cpu().numpy() - ref) / np.linalg.norm(ref))
    assert err <= 1e-10
