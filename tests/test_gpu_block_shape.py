"""FP64 local solves at the numbers of subdomains where the warps per subdomain change (76, 304), by the
preconditioner without the coarse space against the oracle's banded Cholesky (tolerance as in the other
FP64 preconditioner tests)."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver, oracle_problem, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [76, 77, 304, 305])
def test_preconditioner_matches_oracle(L):
    w = Workload("shape", p=1, L=L, n=6, overlap=1, kind="cos1")
    P = oracle_problem(w, coarse=False)
    r = np.random.default_rng(L).standard_normal(w.dofs)
    with make_solver(w, coarse=0) as es:
        es.prepare()
        z = gpu_vec(np.zeros(w.dofs))
        dd.dd_apply_preconditioner(es.ctx, gpu_vec(r), z)
    assert rel_err(host(z), P.prec(r)) < 1e-10
