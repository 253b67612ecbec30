"""phi_s of single-level cells at the factorization's panel, warp and register
edges (16 to 256 nodes, 320 by elimination): each electrode's block solved
exactly, against a dense solve of the oracle's block."""
import numpy as np
import pytest
import torch

from p4d_inputs import make_box_case
from oracle.blocks import BlockPrecond
from oracle.fe import Disc

pytestmark = pytest.mark.gpu

# elements (nx, ny, layers), coarse_max
CASES = {
    "16": (1, 1, (1, 1, 1), 256), "36": (2, 2, (1, 1, 1), 256), "64": (3, 3, (1, 1, 1), 256),
    "75": (2, 4, (1, 1, 2), 256), "128": (3, 7, (1, 1, 1), 256), "160": (3, 7, (1, 1, 2), 256),
    "255": (2, 16, (1, 1, 2), 256), "256": (7, 7, (1, 1, 1), 256), "320": (7, 7, (1, 1, 2), 400),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07225_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(CASES))
def test_phis_of_each_electrode_matches_dense_solve(name):
    from paper_2602_07225_gb300 import P4DSolver
    nx, ny, layers, cm = CASES[name]
    case = make_box_case(nx, ny, layers, 60e-6, (40e-6, 15e-6, 40e-6), 4, 400 + nx)
    d = Disc(case["mesh"], case["params"])
    J = d.jacobian(d.state_from_case(case["state"]))
    s = P4DSolver(case, precision=0, mode=0, coarse_max=cm)
    s.jacobian_update(s.state_tensors(case["state"]))
    A = BlockPrecond(d, J, coarse_max=cm).blocks[0][0].toarray()
    r = np.random.default_rng(23).standard_normal(d.ndof) * np.sqrt(J.diagonal())
    r[3 * d.nn:] = 0.0     # no condensation: phi_s = A_h^-1 r_h
    z = s.precond(torch.tensor(r, device="cuda")).cpu().numpy()
    for e in (0, 1):
        m = np.zeros(d.nn, bool)
        m[d.enodes[d.etype == e]] = True
        m &= d.act
        sc = np.sqrt(np.diag(A)[m])
        B = A[np.ix_(m, m)] / sc[:, None] / sc
        y = np.linalg.solve(B, r[:d.nn][m] / sc)
        # factorization, substitutions and the entries' own rounding: a small
        # multiple of n u in the matrix, times its condition number
        tol = 10 * d.nn * 1.1e-16 * np.linalg.cond(B)
        assert np.linalg.norm(sc * z[:d.nn][m] - y) <= tol * np.linalg.norm(y)
