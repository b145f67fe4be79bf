"""DD_OPT_TILED3 = -1, the default, takes the cached form of the p = 2 float-pair matvec for small boxes and for
cells of few classes, the register-table form for the others: the solves' bits are those of the form the
box calls for."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n,ell,form", [(6, 4, 1.0, 0), (20, 8, 0.5, 0), (10, 16, 0.5, 0), (12, 16, 0.5, 1), (10, 16, 1.0, 1),
                                          (3, 6, 12.0, 0)])
def test_default_form(L, n, ell, form):
    w = Workload("auto", p=2, L=L, n=n, ell=ell, overlap=1, kind="asym3")
    b = gpu_vec(np.random.default_rng(L).standard_normal(w.dofs))
    out = {}
    with make_solver(w, precision="bf16") as es:
        es.prepare()
        for opt in (None, -1, form):
            if opt is not None:
                dd.dd_set_option(es.ctx, dd.DD_OPT_TILED3, opt)
            x = gpu_vec(np.zeros(w.dofs))
            it, rel = dd.dd_pcg_solve(es.ctx, b, x)
            out[opt] = (it, rel, host(x))
        for bad in (-2, 2):
            with pytest.raises(dd.DDError):
                dd.dd_set_option(es.ctx, dd.DD_OPT_TILED3, bad)
    for opt in (-1, form):
        assert out[opt][:2] == out[None][:2] and np.array_equal(out[opt][2], out[None][2])
