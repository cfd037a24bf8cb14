"""Levelled rows of the windowed LU (window_row_scale in csrc/bte_window.cu): calls with two refinement sweeps, on
grids without the FP64 escalation, that the dense LU refined in time and the factors with rows as they come did
not; and FP64 solves that need no correction.

Tolerance against the dense LU, refined with its default sweeps: both stop at max|r| <= refine_tol max|b| (1e-12)
or at a backward error of 256 eps = 2.8e-14; with the condition of the levelled system (below 4e6 on finer grids at
stronger fields than these) the two are within 2 x 4e6 x 2.8e-14 = 2.3e-7."""
import numpy as np
import pytest

from paper_2502_16555_gb300 import workloads as W
from tests._lib import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (workload, nx, nr, ntheta, nl, dt / workload's, |E|, seed)
@pytest.mark.parametrize("case", [("LARGEST", 11, 126, 26, 26, 1.2, 2.84798e5, 111),
                                  ("SMALL", 3, 121, 30, 19, 0.89, 2.9816e4, 195)])
def test_two_sweeps_are_enough_where_they_were_for_the_dense_lu(case):
    from paper_2502_16555_gb300 import bte
    gas, nx, nr, nt, nl, dtf, e0, seed = case
    cfg = W.scaled(getattr(W, gas), nx=nx, nr=nr, ntheta=nt, nl=nl)
    cfg["dt_s"] *= dtf
    F0 = W.random_state(nx, nt, nr, seed=seed + 1)
    E = torch.from_numpy(W.random_field(nx, seed=seed + 2, e0=e0)).cuda()
    out = []
    for kw in (dict(refine_max=2), dict(full_v=True)):
        s = bte.Solver(cfg, precision="mixed", **kw)
        F = torch.from_numpy(F0.copy()).cuda()
        s.step(F, 0.0, E=E)
        out.append(F.cpu().numpy())
    assert float(np.linalg.norm(out[0] - out[1]) / np.linalg.norm(out[1])) <= 2.3e-7


@pytest.mark.parametrize("nr,nt", [(48, 16), (64, 5), (32, 8)])
def test_fp64_solves_need_no_correction(nr, nt):
    """One residual evaluation a point: the first solve's backward error is at rounding level."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.MEDIUM, nx=6, nr=nr, ntheta=nt)
    s = bte.Solver(cfg, precision="fp64")
    F = torch.from_numpy(W.random_state(6, nt, nr, seed=77)).cuda()
    s.step(F, 0.0, E=torch.from_numpy(W.random_field(6, seed=16, e0=4e3)).cuda())
    assert s.info()["last_refine_evals"] == 1.0
