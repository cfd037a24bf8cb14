"""The mixed structured solve with at most one refinement sweep (csrc/bte_struct.cu): its results show the FP32
solve's own accuracy. Unrefined, a step is within 1e-6 of the oracle, twice the largest error (5.2e-7) that the
elimination of the mass-scaled blocks left over 156 grids, fields and states of these sizes."""
import numpy as np
import pytest

from oracle import bte as O
from paper_2502_16555_gb300 import workloads as W
from tests._lib import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("shape", [(32, 8, 8), (48, 16, 16), (64, 5, 4), (21, 8, 1), (17, 6, 3)])
@pytest.mark.parametrize("sweeps", [0, 1])
def test_structured_mixed_step_hardly_refined(shape, sweeps):
    from paper_2502_16555_gb300 import bte
    nr, nt, nl = shape
    cfg = W.scaled(W.MEDIUM, nx=6, nr=nr, ntheta=nt, nl=nl)
    ops = O.Operators(cfg)
    E = W.random_field(6, seed=15, e0=4e3)
    for F0 in (W.random_state(6, nt, nr, seed=75), ops.initial_state()):
        ref = ops.step(F0, 0.0, E=E)
        s = bte.Solver(cfg, precision="mixed", structured=True, refine_max=sweeps)
        F = torch.from_numpy(F0.copy()).cuda()
        s.step(F, 0.0, E=torch.from_numpy(E).cuda())
        err = float(np.linalg.norm(F.cpu().numpy() - ref) / np.linalg.norm(ref))
        assert err <= (1e-6 if sweeps == 0 else 1e-9), err
