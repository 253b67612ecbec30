"""The V-cycle's single-launch tail (one cluster per hierarchy, k_tail) against
the oracle's algorithm at the edges of its rules: one block exactly full, a
few rows into the next block, the largest cluster exactly full, one level too
large for it (level 0 by its own kernels, tail from level 1), and odd sizes;
Chebyshev degrees of both parities, block Jacobi and one block after another."""
import numpy as np
import pytest
import torch

from p4d_inputs import make_box_case
from oracle.blocks import BlockPrecond
from oracle.fe import Disc

pytestmark = pytest.mark.gpu

# elements (nx, ny, layers); nodes
MESHES = {
    "512": (7, 3, (6, 3, 6)),           # 8 x 4 x 16 nodes: one block of 512 rows
    "528": (10, 2, (6, 3, 6)),          # 11 x 3 x 16: 16 rows into the second block
    "4096": (15, 15, (6, 3, 6)),        # 16^3: the FP64 rule's largest level
    "4352": (15, 16, (6, 3, 6)),        # 16 x 17 x 16: above it (FP64 tail from level 1)
    "8192": (31, 15, (6, 3, 6)),        # 32 x 16 x 16: the FP32 rule's largest level
    "9982": (45, 30, (2, 2, 2)),        # 46 x 31 x 7: level 0 matrix-free, last tiles one node wide
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07225_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("precision,combine,cheb", [(1, 0, (2, 10.0)), (1, 1, (3, 20.0)), (0, 0, (1, 4.0)),
                                                    (0, 1, (2, 10.0)), (2, 0, (2, 10.0))])
def test_tail_matches_oracle_algorithm(name, precision, combine, cheb):
    from paper_2602_07225_gb300 import P4DSolver
    nx, ny, layers = MESHES[name]
    case = make_box_case(nx, ny, layers, 60e-6, (40e-6, 15e-6, 40e-6), 4, 1300 + nx)
    d = Disc(case["mesh"], case["params"])
    ref = d.state_from_case(case["state"])
    J = d.jacobian(ref)
    s = P4DSolver(case, precision=precision, combine=combine, mode=0, cheb_degree=cheb[0], cheb_ratio=cheb[1])
    s.jacobian_update(s.state_tensors(case["state"]))
    P = BlockPrecond(d, J, combine="multiplicative" if combine else "additive", order=(1, 0, 2), degree=cheb[0],
                     ratio=cheb[1])
    r = np.random.default_rng(17).standard_normal(d.ndof) * np.sqrt(J.diagonal())
    z = s.precond(torch.tensor(r, device="cuda")).cpu().numpy()
    z_ref = P.apply(r)
    errs = [np.linalg.norm(z[sl] - z_ref[sl]) / np.linalg.norm(z_ref[sl]) for sl in d.field_slices()]
    # the bounds of the same comparisons on the other meshes: FP64 rounding
    # (phi_s, and what follows it, amplified by its near-constant mode), about
    # 170 FP32 unit roundoffs, and one BF16 unit roundoff of the stored levels
    tol = {0: [1e-7, 1e-7 if combine else 1e-11, 1e-7 if combine else 1e-11, 1e-7], 1: [1e-5] * 4, 2: [3e-3] * 4}
    # phi_s (and c_s after it) on the smallest meshes: the near-constant mode
    # of the cathode is anchored by the reaction alone, and its condition
    # number times the unit roundoff passes those bounds whatever the kernel
    # (level by level, FP64: 1.7e-7 on "528"); c_e follows phi_s only there
    fields = (1, 2) if d.nn < 1000 else (0, 1, 2, 3)
    assert all(errs[f] < tol[precision][f] for f in fields), errs
