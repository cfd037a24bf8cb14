"""The structured velocity solve (csrc/bte_struct.cu) at the edges of its 16 x 16 register blocks: one
block short of, at and past each boundary, the widest block, one harmonic (only S_0, not symmetric) and
two. One step from a random state with a field per point against the FP64 oracle.

Tolerances: those of the parity tests, 1e-10 (FP64) and 1e-9 (mixed, refined to a 1e-12 residual)."""
import numpy as np
import pytest

from oracle import bte as O
from paper_2502_16555_gb300 import workloads as W
from tests._lib import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (nx, nr, ntheta, nl)
SHAPES = [(3, 4, 4, 4), (4, 15, 5, 5), (4, 16, 4, 4), (3, 17, 6, 6), (4, 31, 3, 2), (3, 33, 5, 4), (3, 48, 4, 4),
          (3, 49, 8, 8), (3, 64, 3, 1), (3, 64, 40, 40), (160, 18, 3, 3)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_structured_block_edges(shape, precision):
    from paper_2502_16555_gb300 import bte
    nx, nr, nt, nl = shape
    cfg = W.scaled(W.MEDIUM, nx=nx, nr=nr, ntheta=nt, nl=nl)
    ops = O.Operators(cfg)
    F0 = W.random_state(nx, nt, nr, seed=67)
    E = W.random_field(nx, seed=9, e0=8e3)
    E[0] = 0.0
    ref = ops.step(F0, 0.0, E=E)
    F = torch.from_numpy(F0).cuda()
    bte.Solver(cfg, precision=precision, structured=True).step(F, 0.0, E=torch.from_numpy(E).cuda())
    err = float(np.linalg.norm(F.cpu().numpy() - ref) / np.linalg.norm(ref))
    assert err <= (1e-10 if precision == "fp64" else 1e-9)
