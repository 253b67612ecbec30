"""Load and store inside the V-cycle's single launch (reduced block Jacobi of
cells that lie wholly in the tail): one FGMRES step from zero leaves
x = y_0 P^-1 b, compared with p4d_precond_apply, which loads and stores by
launches of their own."""
import numpy as np
import pytest
import torch

from p4d_inputs import make_box_case
from oracle.fe import Disc

pytestmark = pytest.mark.gpu

# elements (nx, ny, layers), lateral size
MESHES = {
    "512": (7, 3, (6, 3, 6), 60e-6), "528": (10, 2, (6, 3, 6), 60e-6), "2025": (8, 8, (10, 4, 10), 100e-6),
    "1953": (8, 6, (8, 10, 12), 0.3e-3), "4096": (15, 15, (6, 3, 6), 60e-6), "8192": (31, 15, (6, 3, 6), 60e-6),
    "4352": (15, 16, (6, 3, 6), 60e-6),      # FP64: level 0 by its own launches
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07225_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("adjoint", [False, True])
def test_one_step_solution_is_the_preconditioned_right_hand_side(name, precision, adjoint):
    from paper_2602_07225_gb300 import P4DSolver
    nx, ny, layers, lat = MESHES[name]
    case = make_box_case(nx, ny, layers, lat, (40e-6, 15e-6, 40e-6), 4, 900 + nx)
    s = P4DSolver(case, precision=precision, mode=1, combine=0, rtol=1e-14, maxit=1)
    st = s.state_tensors(case["state"])
    s.jacobian_update(st)
    nn = s.nn
    # positive at the scale of the rows' diagonals: relative changes of its
    # entries do not grow in the result (the oracle's V-cycle; identity rows keep them);
    # none on the particles, nothing to condense
    d = Disc(case["mesh"], case["params"])
    dg = np.sqrt(d.jacobian(d.state_from_case(case["state"])).diagonal())
    dg[3 * nn:] = 0.0
    b = torch.tensor(np.random.default_rng(31).uniform(0.5, 1.5, s.ndof) * dg, device="cuda")
    x, info = s.solve(b, adjoint=adjoint, check=False)
    assert info["iters"] == 1
    z = s.precond(b, transpose=adjoint)
    x, z = x[:3 * nn].view(3, nn).cpu().numpy(), z[:3 * nn].view(3, nn).cpu().numpy()
    y0 = (x[2] @ z[2]) / (z[2] @ z[2])
    elec = np.full(nn, -1)
    elec[d.enodes] = d.etype
    every = np.ones(nn, bool)
    parts = [(0, ~d.act), (0, d.act & (elec == 0)), (0, d.act & (elec == 1)), (1, every), (2, every)]
    # the scaling and its inverse are FP32 numbers, 6e-8 off each other, which
    # the FP64 path sees as they are; the FP32 load rounds three times more, and
    # the cycle itself to about 170 unit roundoffs (test_gpu_tail)
    tol = 1e-6 if precision == 0 else 1e-5
    errs = [np.linalg.norm(x[f][m] - y0 * z[f][m]) / abs(y0) / np.linalg.norm(z[f][m]) for f, m in parts]
    assert max(errs) <= tol, errs
