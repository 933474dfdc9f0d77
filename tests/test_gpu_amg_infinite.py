"""An iterate that overflows in the AMG V-cycle's levels that run in one
thread-block cluster: a missing neighbour reads as zero whatever the iterates
hold, as in the form with one kernel per half sweep, so the infinity reaches
the same cells in both.  (Its coefficient alone would not do: 0 times an
infinity is NaN.)

The right-hand side is a point source whose solution overflows at the source
in the post-smoothing: its red neighbours then become infinite, all other
cells stay finite."""
import numpy as np
import pytest

import bogen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bo():
    import paper_1606_00556_gb300 as m
    m.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return m


# one block, levels shared by two to sixteen blocks
@pytest.mark.parametrize("dims", [(16, 9, 2), (10, 10, 10), (34, 31, 3), (32, 32, 16)])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_an_overflow_reaches_the_same_cells_as_with_one_kernel_per_half_sweep(bo, dims, precision):
    nx, ny, nz = dims
    N = nx * ny * nz
    a = bogen.assemble(bogen.tiny_case(3, *dims))
    val = a["val"] * 2.0 ** (-10 - np.ceil(np.log2(np.abs(a["val"]).max())))  # (so that the iterates overflow first)
    ctx = bo.Context(0)
    A = bo.Matrix.from_bsr(ctx, bo.grid(*dims), a["rowptr"], a["col"], val)
    P = bo.Preconditioner(A, precision=precision, nu1=1, nu2=1)
    b = 2 * nx - 2  # a black cell of the second row's last pair; the first cell of the third row has no -x neighbour
    top = float(np.finfo(np.float64 if precision == 0 else np.float32).max)

    def apply(mode, source):
        r = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
        r[3 * b] = source
        bo.bo_set_amg_cooperative(mode)
        try:
            return P.apply(bo.BO_STAGE_AMG, r, torch.zeros_like(r))[::3].clone()
        finally:
            bo.bo_set_amg_cooperative(2)

    unit = apply(0, 1.0)
    assert torch.equal(unit, apply(2, 1.0)) and int(unit.argmax()) == b
    z = [apply(mode, 1.02 * (top / float(unit.max()))) for mode in (0, 2)]
    lost = torch.nonzero(~torch.isfinite(z[0])).view(-1).tolist()
    assert lost == [b - nx, b - 1, b, b + 1, b + nx] + ([b + nx * ny] if nz > 1 else []) and not z[0].isnan().any()
    assert torch.equal(z[0], z[1])
    P.close()
