"""Right-hand sides whose squared norm is not a finite number: the solve ends
with the non-finite status (not a CUDA error), the same launched as graphs and
step by step, and the handle solves on."""
import pytest
import torch

from p4d_inputs import make_box_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07225_gb300 import build
    build.build()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("fields", [(0,), (1,), (0, 1, 2)])
def test_overflowing_right_hand_side(mode, adjoint, fields):
    from paper_2602_07225_gb300 import P4DSolver
    from paper_2602_07225_gb300._native import NONFINITE
    case = make_box_case(10, 2, (6, 3, 6), 60e-6, (40e-6, 15e-6, 40e-6), 4, 71)
    s = P4DSolver(case, mode=mode, rtol=1e-8, maxit=200)
    st = s.state_tensors(case["state"])
    s.jacobian_update(st)
    b = -s.residual(st)
    x0, _ = s.solve(b, adjoint=adjoint)
    big = b.clone()
    for f in fields:
        big[f * s.nn:(f + 1) * s.nn] = 1e200     # finite, its square is not
    got = []
    for profile in (1, 0):                       # step by step, as graphs
        s.set_options(profile=profile)
        _, info = s.solve(big, adjoint=adjoint, check=False)
        got.append((info["status"], info["iters"], info["restarts"]))
    assert got[0] == got[1] and got[0][0] == NONFINITE
    x1, _ = s.solve(b, adjoint=adjoint)
    assert torch.equal(x0, x1)
