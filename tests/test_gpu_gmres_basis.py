"""The Gram-Schmidt passes of GMRES over the numbers of basis vectors at which they take another
split of the warps (1 to 8 vectors: several warps each; up to 16: one; more: two vectors per
warp and round) and both forms of the triangular solve (up to 71 columns staged in shared
memory), on boxes of one block with a ragged run and of many blocks."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from oracle import solvers
from tests.gpu_util import gpu_vec, host, make_solver, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n,restart,coarse", [(2, 6, 30, 1), (12, 8, 6, 1), (12, 8, 12, 1), (40, 8, 24, 1), (40, 8, 34, 1),
                                                (60, 8, 71, 0), (60, 8, 72, 0), (60, 8, 200, 0)])
def test_gmres_against_oracle(L, n, restart, coarse):
    w = Workload("basis", p=1, L=L, n=n, overlap=1, kind="cos1")
    P = oracle_problem(w, coarse=bool(coarse))
    b = np.random.default_rng(5).standard_normal(w.dofs)
    _, it_o, _ = solvers.gmres(P.Asig, b, None, P.prec, 1e-8, restart)
    with make_solver(w, coarse=coarse) as es:
        es.prepare()
        dd.dd_set_option(es.ctx, dd.DD_OPT_RESTART, restart)
        x = gpu_vec(np.zeros(w.dofs))
        it, rel = dd.dd_gmres_solve(es.ctx, gpu_vec(b), x, rtol=1e-8)
        assert rel <= 1e-8
        # the counts of restarted cycles follow rounding where the residual stalls (one part in 50)
        assert abs(it - it_o) <= 1 + it_o // 50
        assert np.linalg.norm(b - P.Asig @ host(x)) <= 1.01e-8 * np.linalg.norm(b)
