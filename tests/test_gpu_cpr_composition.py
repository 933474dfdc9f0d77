"""The CPR in FP32 and BF16 storage against the composition it stands for,
  x1 = R^{-1} f,  x2 = x1 + Pi_p AMG(A_pp)^{-1} Pi_r (f - A x1),
  z  = x2 + R^{-1} (f - A x2),
with whole residuals of the rounded decoupled matrix: local solves and
V-cycles by the library's own stages, the residuals here in FP32 in the
matrix's slot order (-z, -y, -x, cell, +x, +y, +z), one fused multiply-add a
product.  Some systems amplify rounding so far that another order of the same
sums moves a solution by more than the solver's tolerance, so the results are
equal bit for bit, in every launch form of the V-cycle.  Sizes: single cells,
rows and planes, odd lengths, several thread blocks."""
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


def _fma32(a, x, acc):
    """a x + acc in one FP32 rounding: the product is exact in FP64, and the
    FP64 sum is rounded to odd before it is rounded to FP32."""
    p, c = a.astype(np.float64) * x, acc.astype(np.float64)
    s = p + c
    bb = s - p
    err = (p - (s - bb)) + (c - bb)
    even = (s.view(np.int64) & 1) == 0
    s = np.where((err != 0) & even, np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return s.astype(np.float32)


def _blocks(Ao, dims, dtype):
    """(7, 3, 3, N) blocks of the decoupled matrix, rounded as the library stores them, and the neighbours (7, N)."""
    At, _ = oracle.qi_decouple(Ao)
    nx, ny, nz = dims
    N = nx * ny * nz
    val = torch.from_numpy(At.val.reshape(-1, 3, 3).astype(np.float32)).to(dtype).float().numpy()
    rows = np.repeat(np.arange(N), np.diff(At.rowptr))
    i, j, k = rows % nx, rows // nx % ny, rows // (nx * ny)
    ci, cj, ck = At.col % nx, At.col // nx % ny, At.col // (nx * ny)
    slot = np.select([ck < k, cj < j, ci < i, ci > i, cj > j, ck > k], [0, 1, 2, 4, 5, 6], 3)
    B = np.zeros((7, 3, 3, N), np.float32)
    nb = np.tile(np.arange(N), (7, 1))
    B[slot, :, :, rows] = val
    nb[slot, rows] = At.col
    return B, nb


def _residual(B, nb, f, x):
    acc = np.zeros_like(f)
    for s in range(7):
        for r in range(3):
            for c in range(3):
                acc[:, r] = _fma32(B[s, r, c], x[nb[s], c], acc[:, r])
    return f - acc


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_cpr_equals_the_whole_residual_composition(bo, dims, storage):
    precision, dtype = {"fp32": (bo.BO_PREC_FP32, torch.float32), "bf16": (bo.BO_PREC_BF16, torch.bfloat16)}[storage]
    a = bogen.assemble(bogen.tiny_case(5, *dims))
    val = a["val"].reshape(-1, 3, 3).copy()
    if storage == "fp32":  # (decoupled rows are formed in 48 bits: FP32 values of them may differ from FP64's)
        val[:, 0, 1:] = 0.0
    ctx = bo.Context(0)
    A = bo.Matrix.from_bsr(ctx, bo.grid(*dims), a["rowptr"], a["col"], val)
    B, nb = _blocks(oracle.BsrMatrix(a["rowptr"], a["col"], val), dims, dtype)
    f = np.random.default_rng(3).standard_normal((B.shape[-1], 3)).astype(np.float32)
    for nu1, nu2 in ((2, 2), (1, 0), (0, 1)):
        P = bo.Preconditioner(A, precision=precision, nu1=nu1, nu2=nu2)

        def stage(st, v):
            r = torch.from_numpy(v.astype(np.float64).ravel()).cuda()
            z = P.apply(st, r, torch.full_like(r, float("nan"))).cpu().numpy().reshape(-1, 3)
            assert np.isfinite(z).all() and np.array_equal(z, z.astype(np.float32))  # FP32 values
            return z.astype(np.float32)

        x1 = stage(bo.BO_STAGE_ILU, f)
        r1 = _residual(B, nb, f, x1)
        for mode in (2, 1, 0):
            bo.bo_set_amg_cooperative(mode)
            try:
                e = stage(bo.BO_STAGE_AMG, r1)
                z = stage(bo.BO_STAGE_CPR_DECOUPLED, f)
            finally:
                bo.bo_set_amg_cooperative(2)
            assert not e[:, 1:].any()
            x2 = x1 + e
            assert np.array_equal(z, x2 + stage(bo.BO_STAGE_ILU, _residual(B, nb, f, x2)))
        P.close()
