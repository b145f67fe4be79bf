"""The register-table form of the p = 2 float-pair matvec (DD_OPT_TILED3 = 1) against the form that
reads the table and p through the caches (0): the same operations per node, so the same bits, at
the shapes where the division into column groups, cells and planes changes: one and several column
groups, a last group with fewer columns, one to five cells along an axis (full and partial sets of
four), the smallest and largest padded column the form takes, and one it leaves to the other."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload
from tests.gpu_util import gpu_vec, host, make_solver

pytestmark = pytest.mark.gpu

CASES = {
    "one_cell": Workload("m", p=2, L=1, n=5, overlap=1, kind="asym3"),
    "two_cells_small_columns": Workload("m", p=2, L=2, n=3, ell=1.0, overlap=1, kind="asym3"),
    "partial_group": Workload("m", p=2, L=3, n=11, overlap=2, kind="asym3"),
    "two_groups": Workload("m", p=2, L=4, n=16, overlap=2, kind="wells"),
    "five_cells": Workload("m", p=2, L=5, n=8, ell=0.5, overlap=1, kind="asym3"),
    "ypad_32": Workload("m", p=2, L=5, n=20, overlap=2, kind="asym3"),
    "ypad_64": Workload("m", p=2, L=3, n=6, ell=6.0, overlap=1, kind="asym3"),
    "ypad_128": Workload("m", p=2, L=2, n=6, ell=12.0, overlap=1, kind="asym3"),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_same_bits_as_the_cached_form(name):
    w = CASES[name]
    x = gpu_vec(np.random.default_rng(5).standard_normal(w.dofs))
    with make_solver(w, precision="bf16") as es:
        dd.dd_cell_eigenpair(es.ctx)
        y = []
        for form in (0, 1):
            dd.dd_set_option(es.ctx, dd.DD_OPT_TILED3, form)
            v = gpu_vec(np.zeros(w.dofs))
            dd.dd_apply_asigma_pairs(es.ctx, x, v)
            y.append(host(v))
    assert np.array_equal(y[0], y[1])
