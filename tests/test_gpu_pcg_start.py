"""PCG starts r_0 = b - A_sigma x_0 with x_0 zero but for one node: the warps whose taps all read zeros leave
their products out.  Boxes whose padded nodes end inside a warp and at a warp's edge, p = 1 and 2,
the one node first, in the middle and last.  A start that missed a product would leave its size in
the residual that is measured from the solution; the steps are the oracle's."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from oracle import solvers
from tests.gpu_util import gpu_vec, host, make_solver, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,L,n,ell", [(1, 1, 3, 1.0), (1, 2, 3, 1.0), (1, 3, 6, 1.0), (1, 11, 3, 1.0), (1, 40, 8, 1.0),
                                       (2, 1, 3, 1.0), (2, 2, 3, 1.0), (2, 3, 5, 0.8)])
@pytest.mark.parametrize("where", [0.0, 0.5, 1.0])
def test_one_node_start(p, L, n, ell, where):
    w = Workload("start", p=p, L=L, n=n, ell=ell, overlap=1, kind="cos1" if p == 1 else "asym3")
    P = oracle_problem(w)
    b = np.random.default_rng(L).standard_normal(w.dofs)
    x0 = np.zeros(w.dofs)
    x0[int(round(where * (w.dofs - 1)))] = 100.0
    r0 = np.linalg.norm(b - P.Asig @ x0)
    _, it_o, _ = solvers.pcg(P.Asig, b, x0, P.prec, 1e-8)
    with make_solver(w) as es:
        es.prepare()
        x = gpu_vec(x0)
        it, rel = dd.dd_pcg_solve(es.ctx, gpu_vec(b), x, rtol=1e-8)
    assert rel <= 1e-8 and abs(it - it_o) <= 1
    # the recursion's residual and the measured one part by rounding, far below 1e-9 of r_0
    assert np.linalg.norm(b - P.Asig @ host(x)) <= 1.1e-8 * r0
