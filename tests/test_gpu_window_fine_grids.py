"""FP64 windows of fine speed grids on both sides of the sizes where the substitution's ring has one stage
left (csrc/bte_window_plan.h): 136 B-splines with 17 to 32 harmonics, 231 with 9 to 16, and the widest.

Tolerances. Steps, against the dense FP64 LU: 1e-9, that of the widest window's mixed test, whose refinement
stops at ten times the residual of FP64. The adjoint identity: 1e-12, the bound at 33 B-splines, times the
ratio of the condition numbers of M_v (6.5e6 / 2.9e5), to which an unrefined solve is exposed. SC and SA
against the dense LU: 14 cond(M_v) eps for the three unrefined solves that the two sides make."""
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


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nr,nt", [(135, 17), (136, 17), (327, 17), (230, 9), (231, 9)])
def test_fine_speed_grids_match_the_dense_lu(nr, nt):
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=3, nr=nr, ntheta=nt)
    F0 = W.random_state(3, nt, nr, seed=71)
    E = W.random_field(3, seed=12, e0=4e3)
    out = []
    for dense in (False, True):
        s = bte.Solver(cfg, precision="fp64", full_v=dense)
        F = torch.from_numpy(F0.copy()).cuda()
        s.step(F, 0.0, E=torch.from_numpy(E).cuda())
        s.run(F, 2, 0.2 / W.RF_FREQ_HZ)
        out.append(F.cpu().numpy())
        del s
    assert rel_l2(out[0], out[1]) <= 1e-9


def test_adjoint_on_a_fine_speed_grid():
    from paper_2502_16555_gb300 import bte
    nx, nt, nr = 3, 17, 136
    cfg = W.scaled(W.SMALL, nx=nx, nr=nr, ntheta=nt)
    F0 = W.random_state(nx, nt, nr, seed=72)
    lam0 = np.random.default_rng(72).standard_normal(F0.shape)
    t = 0.21 / W.RF_FREQ_HZ
    out = []
    for dense in (False, True):
        s = bte.Solver(cfg, precision="fp64", full_v=dense)
        F = torch.from_numpy(F0.copy()).cuda()
        lam = torch.from_numpy(lam0.copy()).cuda()
        SC = torch.zeros((nt * nr, nt * nr), dtype=torch.float64, device="cuda")
        SA = torch.zeros_like(SC)
        s.step_adjoint(F, lam, t, SC=SC, SA=SA)
        s.step(F, t)
        out.append([x.cpu().numpy() for x in (F, lam, SC, SA)])
        del s
    F, lam = out[0][:2]
    scale = float(np.linalg.norm(lam0) * np.linalg.norm(F))
    assert abs(float(np.sum(lam0 * F)) - float(np.sum(lam * F0))) <= 1e-12 * (6.5e6 / 2.9e5) * scale
    for got, ref in zip(out[0][2:], out[1][2:]):
        assert rel_l2(got, ref) <= 1e-8
