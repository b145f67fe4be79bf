"""DD_OPT_FUSE_XR = -1 takes the fused x/r update up to 512 subdomains: the same iterations and bits as
the separate update on both sides of that line, and for the smallest boxes."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "tf32"])
@pytest.mark.parametrize("L", [1, 2, 37, 512, 513])
def test_same_bits_as_the_separate_update(L, precision):
    w = Workload("auto", p=1, L=L, n=6, overlap=2, kind="cos1")
    b = gpu_vec(np.random.default_rng(L).standard_normal(w.dofs))
    out = []
    with make_solver(w, precision=precision) as es:
        es.prepare()
        for opt in (0, -1, 1):
            dd.dd_set_option(es.ctx, dd.DD_OPT_FUSE_XR, opt)
            x = gpu_vec(np.zeros(w.dofs))
            it, _ = dd.dd_pcg_solve(es.ctx, b, x)
            out.append((it, host(x)))
    assert out[0][0] == out[1][0] == out[2][0]
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][1], out[2][1])
