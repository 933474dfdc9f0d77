"""The CPR's passes between its two local solves (no residual formed on the
red cells, the first pre-smoothing sweep and the last post-smoothing half
sweep of the AMG's level 0 folded into them) against the oracle's composition
of whole residuals, local solves and V-cycles: every launch form of the
V-cycle, every number of sweeps, single cells, rows and planes, one-level
hierarchies.  The bounds are those of the stage parity tests; in BF16 storage,
whose distance from the oracle those tests bound at one size, the launch
forms are compared with one another."""
import numpy as np
import pytest

import bogen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = [(2, 1, 1), (2, 3, 43), (16, 9, 1), (14, 11, 7), (34, 31, 16), (62, 45, 19)]


@pytest.fixture(scope="module")
def bo():
    import paper_1606_00556_gb300 as m
    m.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return m


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_cpr_matches_oracle_in_every_launch_form(bo, dims, precision):
    a = bogen.assemble(bogen.tiny_case(5, *dims))
    ctx = bo.Context(0)
    A = bo.Matrix.from_bsr(ctx, bo.grid(*dims), a["rowptr"], a["col"], a["val"])
    Ao = oracle.BsrMatrix(a["rowptr"], a["col"], a["val"])
    r = np.random.default_rng(3).standard_normal(a["b"].size)
    rd = torch.from_numpy(r).cuda()
    for nu1, nu2 in ((2, 2), (1, 1), (1, 0), (0, 1), (3, 2)):
        ref = oracle.cpr_prec(Ao, dims, amg=oracle.AmgParams(nu1=nu1, nu2=nu2)).apply(r)
        P = bo.Preconditioner(A, precision=precision, nu1=nu1, nu2=nu2)
        forms = {}
        for mode in (2, 1, 0):
            bo.bo_set_amg_cooperative(mode)
            try:
                z = P.apply(bo.BO_STAGE_CPR, rd, torch.full_like(rd, float("nan"))).cpu().numpy()
            finally:
                bo.bo_set_amg_cooperative(2)
            forms[mode] = z
            if precision < 2:
                assert np.abs(z - ref).max() <= (1e-12, 1e-5)[precision] * np.abs(ref).max()
        assert np.isfinite(forms[0]).all() and np.array_equal(forms[2], forms[0])
        P.close()
