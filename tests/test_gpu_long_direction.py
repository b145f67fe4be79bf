"""Boxes whose planes hold more unknowns than a block's shared memory can take (7040) are set up with FP64
local solves, and their operators work (the mass matrix on ones: h^2 at the interior of interior rows);
only their set-up of the preconditioner is beyond a test's time."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from tests.gpu_util import gpu_vec, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n,ny", [(1, 3, 7200), (2, 3, 9000), (1, 4, 7043)])
def test_setup_and_mass(L, n, ny):
    import torch
    grid = dd.make_grid(p=1, L=L, n=n, ell=ny / n, overlap=1, precision="fp64")
    V = torch.zeros(n * ny * 4, dtype=torch.float64, device="cuda")
    with dd.Eigensolver(grid, V) as es:
        for k in (0, 4):
            dd.dd_set_option(es.ctx, dd.DD_OPT_LOCAL_RHS, k)
        ones = gpu_vec(np.ones(es.info["ndof"]))
        y = gpu_vec(np.zeros(es.info["ndof"]))
        dd.dd_apply_operator(es.ctx, dd.DD_OP_MASS, ones, y)
        y = host(y).reshape(L * n - 1, ny - 1)
    h = 1.0 / n
    edge = np.full(ny - 1, 1.0)
    edge[[0, -1]] = 5.0 / 6.0
    col = np.full(L * n - 1, 1.0)
    col[0] -= 1.0 / 6.0
    col[-1] -= 1.0 / 6.0
    # 16 products of sizes up to 4/9 h^2 per node: a few roundings of h^2
    assert np.abs(y - h * h * np.outer(col, edge)).max() <= 16 * np.finfo(float).eps * h * h
