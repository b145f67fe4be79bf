"""The 128 x 64 output tile of the local-solve contraction, forced: the same bits as 128 x 256 (every element is
accumulated over K in the same order) where the number of subdomains ends before, at and after a
tile, in one dimension and in three, and K holds an odd number of half stages; the tile that
dd_query reports can be asked for."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "tf32", "fp8"])
@pytest.mark.parametrize("p,L,n", [(1, 1, 6), (1, 66, 6), (1, 67, 6), (1, 131, 6), (1, 40, 16), (2, 4, 4), (2, 9, 4)])
def test_same_bits_as_the_widest_tile(p, L, n, precision):
    w = Workload("t64", p=p, L=L, n=n, overlap=1, kind="cos1" if p == 1 else "asym3")
    r = gpu_vec(np.random.default_rng(L).standard_normal(w.dofs))
    out = {}
    with make_solver(w, precision=precision) as es:
        es.prepare()
        for bn in (256, 64, es.info["gemm_tile_n"]):
            dd.dd_set_option(es.ctx, dd.DD_OPT_GEMM_TILE_N, bn)
            z = gpu_vec(np.zeros(w.dofs))
            dd.dd_apply_preconditioner(es.ctx, r, z)
            out[bn] = host(z)
    assert all(np.array_equal(v, out[256]) for v in out.values())


def test_other_tiles_are_refused():
    with make_solver(Workload("t64", p=1, L=2, n=6, overlap=1, kind="cos1"), precision="bf16") as es:
        for bn in (-64, 1, 32, 96, 512):
            with pytest.raises(dd.DDError):
                dd.dd_set_option(es.ctx, dd.DD_OPT_GEMM_TILE_N, bn)
