"""FP64 local solves by planes (twisted block elimination with dense inverse Schur complements)
against the oracle's banded Cholesky per subdomain, through dd_apply_preconditioner without the
coarse space (whose own conditioning grows like L^2 and would hide the local part), at the sizes
where the kernels change: planes of fewer than, exactly and more than 32 unknowns, one, two and
four warps per subdomain, one, two and four subdomains per block, several blocks per side,
odd and even numbers of planes, one and two subdomains in all.  The tolerance is that of the
other FP64 preconditioner tests (1e-10): both forms are accurate to eps cond(A_i), and the local
condition numbers here are at most a few 1e4."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver, oracle_problem, rel_err

pytestmark = pytest.mark.gpu

CASES = {
    "one_cell": Workload("b", p=1, L=1, n=8, overlap=1, kind="cos1"),
    "two_cells_even": Workload("b", p=1, L=2, n=9, overlap=2, kind="cos1"),
    "rows_1": Workload("b", p=1, L=4, n=4, ell=0.5, overlap=1, kind="cos1"),
    "rows_32": Workload("b", p=1, L=3, n=33, overlap=2, kind="cos4", seed=1),
    "rows_33": Workload("b", p=1, L=3, n=34, overlap=2, kind="cos4", seed=1),
    "rows_95_many": Workload("b", p=1, L=90, n=6, ell=16.0, overlap=1, kind="cos1"),
    "warps_2": Workload("b", p=1, L=100, n=24, overlap=3, kind="cos4", seed=2),
    "block_1": Workload("b", p=1, L=401, n=6, overlap=1, kind="cos1"),
    "block_2": Workload("b", p=1, L=901, n=5, overlap=1, kind="cos1"),
    "block_4": Workload("b", p=1, L=1603, n=4, overlap=1, kind="cos1"),
    "p2_rows_15": Workload("b", p=2, L=3, n=4, overlap=1, kind="asym3"),
    "p2_rows_63": Workload("b", p=2, L=3, n=8, overlap=1, kind="asym3"),
    "p2_sides_4": Workload("b", p=2, L=2, n=15, overlap=2, kind="asym3"),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_preconditioner_matches_oracle(name):
    w = CASES[name]
    P = oracle_problem(w, coarse=False)
    r = np.random.default_rng(3).standard_normal(w.dofs)
    with make_solver(w, coarse=0) as es:
        es.prepare()
        z = gpu_vec(np.zeros(w.dofs))
        dd.dd_apply_preconditioner(es.ctx, gpu_vec(r), z)
        for k in (1, 2, 4):   # subdomains per block: the same bits
            dd.dd_set_option(es.ctx, dd.DD_OPT_LOCAL_RHS, k)
            zk = gpu_vec(np.zeros(w.dofs))
            dd.dd_apply_preconditioner(es.ctx, gpu_vec(r), zk)
            assert np.array_equal(host(zk), host(z))
    assert rel_err(host(z), P.prec(r)) < 1e-10
