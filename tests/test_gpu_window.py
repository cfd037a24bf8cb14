"""The windowed LU of the harmonic system (csrc/bte_window.cu) where its shapes change: unused columns
in a chunk (nl not a power of two), one and several speed indices per chunk, one chunk in all, systems
shorter than the ring, the first far column, a chunk boundary among the far columns, the widest ring
with the most far columns, more points than SMs. One step from a random state with a field per point
against the FP64 oracle and against the dense LU of the same handle kind.

Tolerances: those of the parity tests, 1e-10 (FP64) and 1e-9 (mixed, refined to a 1e-12 residual),
for both comparisons."""
import numpy as np
import pytest

from oracle import bte as O
from paper_2502_16555_gb300 import workloads as W
from tests._lib import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (nx, nr, ntheta, nl); a chunk holds g = 32 / nlp speed indices, nlp the power of two >= nl; the first
# far column is speed index (2 ceil(3 / g) + 1) g
SHAPES = [
    (4, 10, 4, 1),      # g = 32: one chunk
    (4, 70, 3, 1),      # three chunks, no far column
    (3, 130, 3, 1),     # far columns (from 96) behind a ring of two chunks
    (5, 16, 5, 2),      # g = 16: exactly one chunk
    (5, 49, 5, 2),      # one far column
    (4, 33, 7, 3),      # unused column in each group of four; a chunk boundary at 32
    (4, 24, 4, 4),      # all columns used, exactly the ring
    (4, 61, 6, 5),      # g = 4, unused columns
    (3, 9, 17, 16),     # g = 2, shorter than the ring
    (3, 12, 16, 16),    # two far columns
    (3, 45, 17, 17),    # g = 1, 15 unused columns per chunk
    (3, 40, 32, 32),    # far columns 33, just over a chunk of 32
    (3, 7, 32, 32),     # as many chunks as the ring holds
    (160, 8, 5, 5),     # two waves of points
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_window_shapes(shape, precision):
    from paper_2502_16555_gb300 import bte
    nx, nr, nt, nl = shape
    cfg = W.scaled(W.MEDIUM, nx=nx, nr=nr, ntheta=nt, nl=nl)
    ops = O.Operators(cfg)
    F0 = W.random_state(nx, nt, nr, seed=61)
    E = W.random_field(nx, seed=8, e0=8e3)
    E[0] = 0.0
    ref = ops.step(F0, 0.0, E=E)
    tol = 1e-10 if precision == "fp64" else 1e-9
    out = []
    for dense in (False, True):
        s = bte.Solver(cfg, precision=precision, full_v=dense)
        F = torch.from_numpy(F0.copy()).cuda()
        s.step(F, 0.0, E=torch.from_numpy(E).cuda())
        out.append(F.cpu().numpy())
        assert rel_l2(out[-1], ref) <= tol, dense
    assert rel_l2(out[0], out[1]) <= tol


@pytest.mark.parametrize("nr,nt", [(320, 17), (544, 2)])
def test_window_widest(nr, nt):
    """512 window columns: nr = 320 with 17 harmonics; 544 is past the limit for two harmonics (a ring of
    64 columns and 496 far ones) and takes the dense LU. Mixed precision against the dense FP64 LU."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=3, nr=nr, ntheta=nt)
    F0 = W.random_state(3, nt, nr, seed=62)
    out = []
    for precision, dense in (("mixed", False), ("fp64", True)):
        s = bte.Solver(cfg, precision=precision, full_v=dense)
        F = torch.from_numpy(F0.copy()).cuda()
        s.step(F, 0.2 / W.RF_FREQ_HZ)
        out.append(F.cpu().numpy())
        del s
    assert rel_l2(out[0], out[1]) <= 1e-9


def test_adjoint_identity_through_the_window():
    """<lambda, S F> = <S^T lambda, F> to 1e-12 (the bound of the dense transposed solve's test) on a grid
    with unused columns and far columns."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=7, nr=33, ntheta=11)
    rng = np.random.default_rng(63)
    F0 = W.random_state(7, 11, 33, seed=63)
    lam0 = rng.standard_normal(F0.shape)
    t = 0.21 / W.RF_FREQ_HZ
    s = bte.Solver(cfg, precision="fp64")
    F = torch.from_numpy(F0.copy()).cuda()
    lam = torch.from_numpy(lam0.copy()).cuda()
    s.step_adjoint(F, lam, t)
    s.step(F, t)
    a = float(np.sum(lam0 * F.cpu().numpy()))
    b = float(np.sum(lam.cpu().numpy() * F0))
    scale = float(np.linalg.norm(lam0) * np.linalg.norm(F.cpu().numpy()))
    assert abs(a - b) <= 1e-12 * scale, (a, b, scale)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_unfactorable_and_nonfinite_fields_through_the_window(precision):
    """A field that overflows the factors at one point reports BTE_ESINGULAR, a NaN BTE_ENONFINITE; the state
    is kept and the handle steps normally afterwards (nl = 5: several chunks with unused columns)."""
    from paper_2502_16555_gb300 import bte
    cfg = W.scaled(W.SMALL, nx=6, nr=21, ntheta=5)
    F0 = W.random_state(6, 5, 21, seed=64)
    s = bte.Solver(cfg, precision=precision)
    F = torch.from_numpy(F0.copy()).cuda()
    for bad, status in ((1e43 if precision == "mixed" else 1e308, (bte.ESINGULAR,)), (np.nan, (bte.ENONFINITE,))):
        E = np.full(6, 1e3)
        E[2] = bad
        with pytest.raises(bte.BteError) as e:
            s.step(F, 0.0, E=torch.from_numpy(E).cuda())
        assert e.value.status in status
        assert np.array_equal(F.cpu().numpy(), F0)
    E[2] = 1e3
    s.step(F, 0.0, E=torch.from_numpy(E).cuda())
    assert rel_l2(F.cpu().numpy(), O.Operators(cfg).step(F0, 0.0, E=E)) <= 1e-9
