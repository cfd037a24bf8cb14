"""A device wait that runs out in the windowed and the structured solves (BTE_FLAG_DIAG_HARMONIC_TIMEOUT: about
1 ms, on a barrier that nothing signals, with copies and products in flight) is reported as BTE_ECUDA by every
entry point that uses their results."""
import time

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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("structured", [False, True])
def test_step_reports_an_expired_wait_and_keeps_the_state(precision, structured):
    """Several panels and far columns (nr = 48, nl = 17). The handle's own second step and a batch's report it too;
    a handle without the flag then steps to the oracle's result."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=5, nr=48, ntheta=17)
    F0 = W.random_state(5, 17, 48, seed=73)
    t = 0.2 / W.RF_FREQ_HZ
    E = torch.from_numpy(W.random_field(5, seed=13, e0=4e3)).cuda()
    s = bte.Solver(cfg, precision=precision, structured=structured, diag_harmonic_timeout=True)
    F = torch.from_numpy(F0.copy()).cuda()
    for call in (lambda: s.step(F, t, E=E), lambda: s.run(F, 2, t), lambda: bte.Batch([s]).run([F], 1, t)):
        t0 = time.perf_counter()
        with pytest.raises(bte.BteError) as e:
            call()
        assert e.value.status == bte.ECUDA
        assert time.perf_counter() - t0 < 2.0  # no wait ran to its own limit
        assert np.array_equal(F.cpu().numpy(), F0)
    del s
    torch.cuda.synchronize()
    bte.Solver(cfg, precision=precision, structured=structured).step(F, t, E=E)
    ref = O.Operators(cfg).step(F0, t, E=E.cpu().numpy())
    err = float(np.linalg.norm(F.cpu().numpy() - ref) / np.linalg.norm(ref))
    assert err <= (1e-10 if precision == "fp64" else 1e-9)


def test_adjoint_reports_an_expired_wait():
    """F* of an expired substitution is no solution: the sensitivities must not come back as good."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=5, nr=20, ntheta=9)
    s = bte.Solver(cfg, precision="fp64", diag_harmonic_timeout=True)
    F = torch.from_numpy(W.random_state(5, 9, 20, seed=74)).cuda()
    lam = torch.ones_like(F)
    SC = torch.zeros((180, 180), dtype=torch.float64, device="cuda")
    with pytest.raises(bte.BteError) as e:
        s.step_adjoint(F, lam, 0.2 / W.RF_FREQ_HZ, SC=SC)
    assert e.value.status == bte.ECUDA
    assert "wait expired" in str(e.value)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_implicit_step_stops_at_an_expired_wait(precision):
    """Its first step already meets the expired wait: no Newton iteration may follow (each Krylov iteration would
    wait again). The semi-implicit step launches fewer than 100 kernels here."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=5, nr=12, ntheta=6)
    s = bte.Solver(cfg, precision=precision, diag_harmonic_timeout=True)
    F = s.initial_state()
    F0 = F.clone()
    ni = torch.full((5,), 1e15, dtype=torch.float64, device="cuda")
    before = s.info()["launches"]
    with pytest.raises(bte.BteError) as e:
        s.step_implicit(F, ni, 0.0)
    assert e.value.status == bte.ECUDA
    assert torch.equal(F, F0)
    assert s.info()["launches"] - before < 100
