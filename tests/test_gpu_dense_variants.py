"""The dense LU's variants, reached with full_v (a handle without flags takes the windowed LU): the batch
autotuner's trials, the step graph across a variant change, the tensor-core trailing update and its panels in
pairs, the transposed solve. Tolerances: those of the parity, batch and adjoint tests of the same comparisons."""
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


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def to_dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("precision,trials", [("mixed", 8), ("fp64", 2)])
def test_autotuner_times_the_variants_of_dense_handles(precision, trials):
    """One trial is three steps of at least ten launches; a windowed handle in the same batch gets none."""
    from paper_2502_16555_gb300 import bte
    cfgs = [W.scaled(W.SMALL, nx=9, nr=16, ntheta=16, p_Torr=0.3, V0=120.0),
            W.scaled(W.SMALL, nx=12, nr=24, ntheta=16, p_Torr=1.5, V0=200.0)]
    sv = [bte.Solver(c, precision, full_v=True) for c in cfgs] + [bte.Solver(cfgs[0], precision)]
    batch = bte.Batch(sv, autotune=True)
    n = [s.info()["launches"] for s in sv]
    assert min(n[:2]) >= trials * 3 * 10 and n[2] == 0, n
    F0 = [W.random_state(c["nx"], c["ntheta"], c["nr"], seed=50 + k) for k, c in enumerate(cfgs)]
    Fs = [to_dev(f) for f in F0 + F0[:1]]
    t0 = 0.17 / W.RF_FREQ_HZ
    batch.run(Fs, 1, t0)
    for k, F in enumerate(Fs):
        ref = O.Operators(cfgs[k % 2]).step(F0[k % 2], t0)
        assert rel_l2(F.cpu().numpy(), ref) <= (1e-10 if precision == "fp64" else 1e-9)
    batch.close()


def test_run_graph_follows_a_change_of_the_dense_variant():
    """Three handles that start in different variants of one shape: the autotuner's choice changes at least one
    of them, and bte_run, whose graph was captured before, then equals the steps launched kernel by kernel."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=6, nr=24, ntheta=16)
    F0 = W.random_state(6, 16, 24, seed=52)
    changed = 0
    for kw, start in (({}, (1, 1, 2)), ({"tc_one_cta": True}, (1, 1, 1)), ({"tc_single": True}, (1, 0, 2))):
        s = bte.Solver(cfg, "mixed", full_v=True, **kw)
        s.run(to_dev(F0), 2, 0.0)
        b = bte.Batch([s], autotune=True)
        i = b.info(0)
        changed += (i["tensor_cores"], i["tc_pair"], i["tc_cg"]) != start
        b.close()
        A, B = to_dev(F0), to_dev(F0)
        s.run(A, 3, 0.0)
        s.profile_start()
        for k in range(3):
            s.step(B, k * cfg["dt_s"])
        s.profile_stop()
        assert torch.equal(A, B)
    assert changed


@pytest.mark.parametrize("shape", [(4, 32, 8), (6, 24, 16), (5, 40, 13), (4, 64, 12), (3, 36, 20)])
def test_dense_tensor_core_update_against_oracle_and_its_variants(shape):
    """nv = 256 to 768: one trailing update up to three in pairs, ragged last panels among them."""
    from paper_2502_16555_gb300 import bte
    nx, nr, nt = shape
    cfg = W.scaled(W.SMALL, nx=nx, nr=nr, ntheta=nt)
    cfg["V0"] = 400.0
    F0 = W.random_state(nx, nt, nr, seed=31)
    t = 0.21 / W.RF_FREQ_HZ
    ref = O.Operators(cfg).step(F0, t)
    for kw in ({}, {"tc_single": True}, {"tc_one_cta": True}, {"panel_tc": True}, {"simt_gemm": True}):
        s = bte.Solver(cfg, "mixed", full_v=True, **kw)
        assert s.info()["tensor_cores"] == (0 if "simt_gemm" in kw else 1)
        F = to_dev(F0)
        s.step(F, t)
        assert rel_l2(F.cpu().numpy(), ref) <= 1e-9, kw


def test_dense_step_adjoint_is_the_transpose():
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.ADJOINT, nx=9, nr=11, ntheta=7)
    s = bte.Solver(cfg, "fp64", full_v=True)
    rng = np.random.default_rng(3)
    F, lam = to_dev(rng.standard_normal((9, 7, 11))), to_dev(rng.standard_normal((9, 7, 11)))
    t = 0.37 / W.RF_FREQ_HZ
    SF, StL = F.clone(), lam.clone()
    s.step(SF, t)
    s.step_adjoint(F, StL, t)
    a, b = float(torch.sum(lam * SF)), float(torch.sum(StL * F))
    assert abs(a - b) <= 1e-12 * (abs(a) + abs(b)), (a, b)
