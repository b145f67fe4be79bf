"""The FP32 band factors by panels of eight columns, at the bands where the kernel takes another
shape (rows of a panel per lane, entries per thread; the cell band is 2 ny - 1, the local one ny):
the preconditioner with TF32 local inverses against the FP64 one, and the steps of the cell solve,
which the factored shift-and-invert preconditions.  Orders are not multiples of eight."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from tests.gpu_util import gpu_vec, host

pytestmark = pytest.mark.gpu


# steps: ln 1e12 / -ln((1 - sqrt x) / (1 + sqrt x)) + 10 with x = (l2 - l1) / (l2 - min V + 1) of the cell
# pencil's two lowest eigenvalues (dense, in FP64): the bound of preconditioned CG for an exact
# shift-and-invert
@pytest.mark.parametrize("ny,steps", [(2, 35), (3, 28), (9, 27), (28, 53), (29, 50), (32, 59), (33, 55), (44, 62), (45, 63), (46, 81), (56, 80), (57, 104), (80, 168)])
def test_tf32_preconditioner_and_cell_steps(ny, steps):
    import torch
    n, L = 6, 3
    V = np.random.default_rng(ny).uniform(0.0, 20.0, n * ny * 4)
    out, sigma = {}, {}
    for precision in ("fp64", "tf32"):
        grid = dd.make_grid(p=1, L=L, n=n, ell=ny / n, overlap=1, precision=precision)
        with dd.Eigensolver(grid, torch.from_numpy(V).cuda()) as es:
            sigma[precision] = es.prepare()
            assert es.info["cell_iters"] <= steps
            r = gpu_vec(np.random.default_rng(1).uniform(0.5, 1.5, es.info["ndof"]))
            z = torch.zeros_like(r)
            dd.dd_apply_preconditioner(es.ctx, r, z)
            out[precision] = host(z)
    assert sigma["tf32"] == pytest.approx(sigma["fp64"], rel=1e-11)
    # entries of the inverses and of r rounded to 11 bits, products of one sign up to the potential's
    # wiggle: 2 * 2^-11 and the FP32 factor's own error, far below it
    assert np.abs(out["tf32"] - out["fp64"]).max() <= 2 * 2.0 ** -11 * np.abs(out["fp64"]).max()
