"""Cells of many thin node planes (the transfers between levels go plane by
plane): more planes than a grid's y extent (65,535), planes that share a block."""
import numpy as np
import pytest
import torch

from p4d_inputs import make_box_case
from oracle.blocks import BlockPrecond
from oracle.fe import Disc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07225_gb300 import build
    build.build()


# elements (nx, ny, layers), thickness
MESHES = {
    "66001 x 4": (1, 1, (30000, 6000, 30000), (0.4, 0.08, 0.4)),
    "2651 x 25": (4, 4, (1300, 50, 1300), (16e-3, 6e-4, 16e-3)),  # ten planes per block, the last ones fewer
    "1051 x 100": (9, 9, (500, 50, 500), (4e-3, 4e-4, 4e-3)),     # two
    "142 x 126": (13, 8, (60, 21, 60), (100e-6, 25e-6, 100e-6)),
    "142 x 128": (31, 3, (60, 21, 60), (100e-6, 25e-6, 100e-6)),  # blocks of one plane
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(MESHES))
def test_preconditioner_matches_oracle_algorithm(name, precision):
    from paper_2602_07225_gb300 import P4DSolver
    nx, ny, layers, thick = MESHES[name]
    case = make_box_case(nx, ny, layers, 60e-6, thick, 3, 5)
    d = Disc(case["mesh"], case["params"])
    J = d.jacobian(d.state_from_case(case["state"]))
    s = P4DSolver(case, precision=precision, mode=0)
    s.jacobian_update(s.state_tensors(case["state"]))
    r = np.random.default_rng(1).standard_normal(d.ndof) * np.sqrt(J.diagonal())
    z = s.precond(torch.tensor(r, device="cuda")).cpu().numpy()
    z_ref = BlockPrecond(d, J).apply(r)
    # phi_e and c_e (the oracle's phi_s smooths over another interval): relative
    # changes of the operator move them up to 80 times as much
    for sl in d.field_slices()[1:3]:
        assert np.linalg.norm(z[sl] - z_ref[sl]) < {0: 1e-11, 1: 1e-5}[precision] * np.linalg.norm(z_ref[sl])


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 4000), (4, 4, 2300), (15, 15, 226)])
def test_tile_depth_of_thin_cells_leaves_the_results(nx, ny, nz):
    """The depth picked for mf_zchunk = 0 (8 planes, 8 and 2 here) and both set by number."""
    from paper_2602_07225_gb300 import P4DSolver
    n = 4 * nz // 9
    case = make_box_case(nx, ny, (n, nz - 2 * n, n), 60e-6, (3e-6 * n, 3e-6 * (nz - 2 * n), 3e-6 * n), 3, 5)
    z = []
    for zc in (0, 2, 8):
        s = P4DSolver(case, precision=1, mf_zchunk=zc)
        s.jacobian_update(s.state_tensors(case["state"]))
        r = torch.tensor(np.random.default_rng(2).standard_normal(s.ndof), device="cuda")
        z.append(s.precond(r))
    assert bool(torch.isfinite(z[0]).all()) and torch.equal(z[0], z[1]) and torch.equal(z[0], z[2])
