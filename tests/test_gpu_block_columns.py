"""FP64 local solves and the columns their products leave out.  Planes of at most 28 unknowns with one
warp per subdomain, and of at most 16 with one per pair of them, end inside a group of four
columns.  For planes of more than 32 unknowns the products run over the chunks of eight columns that
the widest plane has, which divide unevenly among one, two and four ranges (by the number of
subdomains), and the narrower types of a three-dimensional box end inside a range.  Against the
oracle without the coarse space (tolerance as in the other FP64 preconditioner tests)."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver, oracle_problem, rel_err

pytestmark = pytest.mark.gpu

CASES = [(1, L, 4, (m + 1) / 4) for m in (33, 40, 41, 57, 63) for L in (3, 400)]
CASES += [(1, 200, 4, 42 / 4), (1, 300, 4, 42 / 4), (1, 60, 4, 70 / 4), (1, 150, 4, 70 / 4)]
CASES += [(1, 310, 4, (m + 1) / 4) for m in (1, 2, 3, 4, 13, 15, 16, 17, 27, 28, 29, 32)]   # one warp per subdomain or pair
CASES += [(1, L, 4, 1.0) for L in (305, 1300, 3101)]   # pairs: two, four and eight subdomains per block
CASES += [(2, 3, 5, 8 / 5), (2, 3, 5, 12 / 5), (2, 6, 5, 12 / 5), (2, 10, 5, 8 / 5)]


@pytest.mark.parametrize("p,L,n,ell", CASES)
def test_preconditioner_matches_oracle(p, L, n, ell):
    w = Workload("cols", p=p, L=L, n=n, ell=ell, overlap=1, kind="cos1" if p == 1 else "asym3")
    P = oracle_problem(w, coarse=False)
    r = np.random.default_rng(L).standard_normal(w.dofs)
    with make_solver(w, coarse=0) as es:
        es.prepare()
        z = gpu_vec(np.zeros(w.dofs))
        dd.dd_apply_preconditioner(es.ctx, gpu_vec(r), z)
    assert rel_err(host(z), P.prec(r)) < 1e-10
