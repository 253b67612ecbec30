"""The first residual of a solve (the product with an all-zero guess is left
out) and entries that are not finite (they reach the rows of their own 27
neighbours only, also at the faces of the grid)."""
import numpy as np
import pytest
import torch

from p4d_inputs import make_box_case

pytestmark = pytest.mark.gpu

MESHES = {
    "528": (10, 2, (6, 3, 6)),          # 11 x 3 x 16 nodes: below the rule's 8,192
    "8192": (31, 15, (6, 3, 6)),        # 32 x 16 x 16: its last small size
    "9982": (45, 30, (2, 2, 2)),        # 46 x 31 x 7: above it, ragged blocks
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07225_gb300 import build
    build.build()


def _solver(name, **opts):
    from paper_2602_07225_gb300 import P4DSolver
    nx, ny, layers = MESHES[name]
    case = make_box_case(nx, ny, layers, 60e-6, (40e-6, 15e-6, 40e-6), 4, 700 + nx)
    s = P4DSolver(case, **opts)
    st = s.state_tensors(case["state"])
    s.jacobian_update(st)
    nodes = (nx + 1, ny + 1, sum(layers) + 1)
    return s, st, nodes


@pytest.mark.parametrize("name", ["8192", "9982"])
@pytest.mark.parametrize("adjoint", [False, True])
def test_solve_from_zero_and_from_one_nonzero_entry(name, adjoint):
    s, st, nodes = _solver(name, rtol=1e-9, maxit=400)
    nn = int(np.prod(nodes))
    b = -s.residual(st)
    x, info = s.solve(b, adjoint=adjoint)
    assert info["iters"] > 0
    for idx in (nn, 2 * nn + nn // 2, 3 * nn - 1):
        g = torch.zeros_like(b)
        f = slice(idx // nn * nn, idx // nn * nn + nn)
        g[idx] = 10 * x[f].abs().max()
        y, _ = s.solve(b, x=g.clone(), adjoint=adjoint)
        # a guess that was taken for zero would stay in the result as it is
        assert abs(float(y[idx] - x[idx])) < 0.01 * float(g[idx])
    s.set_options(rtol=1e-6)
    y, info = s.solve(b, x=x.clone(), adjoint=adjoint)
    assert info["iters"] == 0 and torch.equal(x[:3 * nn], y[:3 * nn])


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_entry_stays_in_its_neighbourhood(name, transpose, bad):
    s, st, (nx, ny, nz) = _solver(name)
    nn = nx * ny * nz
    k, j, i = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    rng = np.random.default_rng(5)
    x = torch.tensor(rng.standard_normal(s.ndof), device="cuda")
    for (ci, cj, ck) in [(0, 0, 0), (nx - 1, ny - 1, nz - 1), (0, 1, nz // 2), (nx - 1, 0, nz // 2)]:
        near = ((abs(i - ci) <= 1) & (abs(j - cj) <= 1) & (abs(k - ck) <= 1)).reshape(-1)
        far = torch.tensor(np.flatnonzero(~near), device="cuda")
        n = ci + nx * (cj + ny * ck)
        for f in range(3):
            x0, x1 = x.clone(), x.clone()
            x0[f * nn + n], x1[f * nn + n] = 0.0, bad
            y0, y1 = s.jvp(x0, transpose=transpose), s.jvp(x1, transpose=transpose)
            for g in range(3):
                a, c = y0[g * nn:(g + 1) * nn][far], y1[g * nn:(g + 1) * nn][far]
                # 27 products per sum: at most 30 roundings of the largest row
                assert bool(torch.isfinite(c).all())
                assert float((a - c).abs().max()) <= 30 * 2.3e-16 * float(a.abs().max())
    if not transpose:
        # phi_e of a separator node on a face
        near = ((i <= 1) & (abs(j - 1) <= 1) & (abs(k - nz // 2) <= 1)).reshape(-1)
        far = torch.tensor(np.flatnonzero(~near), device="cuda")
        r0 = s.residual(st)
        st["phie"].reshape(-1)[nx * (1 + ny * (nz // 2))] = bad
        r1 = s.residual(st)
        for g in range(3):
            assert torch.equal(r0[g * nn:(g + 1) * nn][far], r1[g * nn:(g + 1) * nn][far])
