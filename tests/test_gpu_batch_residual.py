"""A batch adds up (r, r) of the PCG stop test as the single calls do, bit for bit, so that its
iteration counts cannot part from theirs where a residual meets the tolerance exactly: boxes whose
single solves fuse the x/r update into the packing (up to 512 subdomains) and one whose do not, in
one group, with the default options, with the fused update off and on, and with the x update of
the same iteration (DD_OPT_X_LAG = 0)."""
import numpy as np
import pytest

import paper_2311_08757_gb300 as dd
from ddinputs import Workload, sample_cell_qp
from tests.gpu_util import gpu_vec, host

pytestmark = pytest.mark.gpu


def _ws(lengths):
    return [Workload("br", p=1, L=L, n=6, overlap=2, kind="cos4", seed=L) for L in lengths]


@pytest.mark.parametrize("precision", ["bf16", "tf32"])
@pytest.mark.parametrize("fuse,lag,lengths", [(-1, 1, (3, 4, 37, 300, 512, 513)), (-1, 0, (3, 37, 513)), (-1, 1, (5, 64)),
                                              (-1, 1, (600, 700)), (0, 1, (37, 300)), (1, 1, (37, 600))])
def test_residual_bits(fuse, lag, lengths, precision):
    import torch
    ws = _ws(lengths)
    grids = [dd.grid_from_workload(w, precision=dd.PRECISIONS[precision]) for w in ws]
    Vs = [torch.from_numpy(sample_cell_qp(w)).cuda() for w in ws]
    phis = [gpu_vec(np.zeros(w.dofs)) for w in ws]

    def options(ctx):
        dd.dd_set_option(ctx, dd.DD_OPT_FUSE_XR, fuse)
        dd.dd_set_option(ctx, dd.DD_OPT_X_LAG, lag)

    with dd.Batch(grids, Vs) as b:
        b.set_groups(1)
        for i in range(len(ws)):
            options(b.context(i))
        res = b.ground_states("ipm", phi=phis)
        assert b.info()["last_batched"] == 1
        batch = [dd.dd_pcg_residual(b.context(i)) for i in range(len(ws))]
    for i, w in enumerate(ws):
        with dd.Eigensolver(grids[i], Vs[i]) as es:
            es.prepare()
            options(es.ctx)
            x = gpu_vec(np.ones(w.dofs))
            lam, outer, tot, _ = dd.dd_inverse_iterate(es.ctx, x)
            assert dd.dd_pcg_residual(es.ctx) == batch[i], w.L
        assert (lam, outer, tot) == (res["lambda"][i], res["outer"][i], res["inner"][i])
        assert np.array_equal(host(x), host(phis[i]))
