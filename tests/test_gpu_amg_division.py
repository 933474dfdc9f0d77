"""The FP64 Gauss-Seidel sweeps divide by the diagonal as an FP64 division
does, whatever they keep of it.  The last half sweep of a V-cycle writes the
red cells of level 0 from the black ones that the result holds, so its
arithmetic can be repeated exactly: six fused multiply-adds in the order -z,
-y, -x, +x, +y, +z and a quotient, each rounded once."""
from fractions import Fraction

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


# level 0 in the cluster; above it (legs or one kernel per half sweep)
@pytest.mark.parametrize("dims", [(14, 11, 7), (34, 31, 20)])
@pytest.mark.parametrize("mode", [2, 1, 0])
def test_red_cells_are_rounded_quotients(bo, dims, mode):
    nx, ny, nz = dims
    N = nx * ny * nz
    a = bogen.assemble(bogen.tiny_case(3, *dims))
    val = a["val"].reshape(-1, 3, 3).copy()
    val[:, 0, 1:] = 0.0  # (the decoupled pressure rows are then the matrix's own)
    ctx = bo.Context(0)
    A = bo.Matrix.from_bsr(ctx, bo.grid(*dims), a["rowptr"], a["col"], val)
    P = bo.Preconditioner(A)
    f = np.random.default_rng(4).standard_normal((N, 3))
    bo.bo_set_amg_cooperative(mode)
    try:
        z = P.apply(bo.BO_STAGE_AMG, torch.from_numpy(f.ravel()).cuda(), torch.zeros(3 * N, dtype=torch.float64, device="cuda"))
    finally:
        bo.bo_set_amg_cooperative(2)
    z = z.cpu().numpy()[::3]
    rowptr, col = np.asarray(a["rowptr"]), np.asarray(a["col"])
    cells = [c for c in range(N) if (c % nx + c // nx % ny + c // (nx * ny)) % 2 == 0]
    for c in cells[:: max(1, len(cells) // 400)]:
        s, d = float(f[c, 0]), None
        for e in range(rowptr[c], rowptr[c + 1]):  # (columns ascend: the slot order)
            if col[e] == c:
                d = val[e, 0, 0]
            else:
                s = float(Fraction(s) - Fraction(float(val[e, 0, 0])) * Fraction(float(z[col[e]])))
        assert z[c] == float(Fraction(s) / Fraction(float(d))), c
    P.close()
