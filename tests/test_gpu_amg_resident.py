"""The AMG levels that run in one thread-block cluster (the default launch
form) against one kernel per half sweep: the same arithmetic in the same
order, so the results are equal bit for bit.  Sizes at the edges of the
form: one block, every cluster size, odd lengths (pairs of cells across rows
and planes), the largest level the cluster takes and one above it, coarsest
levels of 1 to 128 cells."""
import numpy as np
import pytest

import bogen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = [(16, 9, 1), (2, 3, 43), (10, 10, 10), (14, 11, 7), (32, 32, 2), (34, 31, 3), (62, 45, 5), (32, 32, 16),
        (34, 31, 16), (32, 32, 32), (34, 32, 31), (62, 45, 19)]


@pytest.fixture(scope="module")
def bo():
    import paper_1606_00556_gb300 as m
    m.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return m


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_cluster_form_equals_one_kernel_per_half_sweep(bo, dims, precision):
    a = bogen.assemble(bogen.tiny_case(3, *dims))
    ctx = bo.Context(0)
    A = bo.Matrix.from_bsr(ctx, bo.grid(*dims), a["rowptr"], a["col"], a["val"])
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(a["b"].size)).cuda()
    for nu1, nu2 in ((2, 2), (1, 3)):
        P = bo.Preconditioner(A, precision=precision, nu1=nu1, nu2=nu2)
        z = []
        for mode in (2, 0):
            bo.bo_set_amg_cooperative(mode)
            try:
                z.append(P.apply(bo.BO_STAGE_AMG, r, torch.full_like(r, float("nan"))).clone())
            finally:
                bo.bo_set_amg_cooperative(2)
        assert torch.isfinite(z[0]).all() and torch.equal(z[0], z[1])
        P.close()
