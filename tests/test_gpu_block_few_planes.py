"""FP64 local solves of boxes with two or three node planes in all and at most 32 unknowns per plane: the
right block of a subdomain's pair then has no product of its own, or one, so its first arrival at
the meeting barrier follows the start of the kernel at once.  Every application gives the same
bits, and the oracle's (tolerance as in the other FP64 preconditioner tests)."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver, oracle_problem, rel_err

pytestmark = pytest.mark.gpu

CASES = {
    "two_planes": Workload("f", p=1, L=1, n=3, overlap=1, kind="cos1"),
    "two_planes_rows_32": Workload("f", p=1, L=1, n=3, ell=11.0, overlap=1, kind="cos1"),
    "three_planes": Workload("f", p=1, L=1, n=4, overlap=1, kind="cos1"),
    "three_and_four_planes": Workload("f", p=1, L=500, n=3, overlap=1, kind="cos1"),
    "p2_two_planes": Workload("f", p=2, L=1, n=3, overlap=1, kind="asym3"),
    "p2_three_planes": Workload("f", p=2, L=2, n=3, overlap=1, kind="asym3"),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_repeated_applications_match_oracle(name):
    w = CASES[name]
    P = oracle_problem(w, coarse=False)
    r = np.random.default_rng(3).standard_normal(w.dofs)
    with make_solver(w, coarse=0) as es:
        es.prepare()
        rv = gpu_vec(r)
        first = None
        for _ in range(50):
            z = gpu_vec(np.zeros(w.dofs))
            dd.dd_apply_preconditioner(es.ctx, rv, z)
            zh = host(z)
            first = zh if first is None else first
            assert np.array_equal(zh, first)
    assert rel_err(first, P.prec(r)) < 1e-10
