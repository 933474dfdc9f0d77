"""Infinities in the tcgen05 weight gradient: they reach the weights whose sum
has a term with them, and no others.  Tiles that reach beyond the grid multiply
zeros there, which an infinite neighbour would turn into NaN.  The reference is
the definition in FP64 with zeros around the grid (so an infinite dY at the
border does give NaN in the taps that lead out of it)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1606_00556_gb300 as bo  # noqa: E402
from oracle import cnn as O  # noqa: E402

LAYERS = [(16, 32), (32, 32), (32, 16)]
# whole tiles; ragged along x, y and both, by one voxel and by more
DIMS = [(64, 8, 2), (24, 8, 4), (33, 6, 3), (16, 5, 2), (7, 3, 1)]


@pytest.fixture
def ctx():
    bo.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    bo.bo_set_conv_engine(1)
    yield bo.Context(0)
    assert bo.bo_tc_status() == bo.BO_OK


def _grads(ctx, dims, x, dy):
    cin, cout = x.shape[2], dy.shape[2]
    dw = torch.full((27, cout, cin), 7.0, device="cuda")
    db = torch.full((cout,), 7.0, device="cuda")
    bo.bo_conv3d_backward_weights(ctx, dims, x, dy, dw, db)
    return dw.double().cpu().numpy(), db.double().cpu().numpy()


def _same(got, ref, mag):
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(got[inf], ref[inf])
    ok = np.isfinite(ref)
    assert (np.abs(got[ok] - ref[ok]) <= 1e-5 * mag[ok] + 1e-30).all()  # (FP32 accumulation)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("cin,cout", LAYERS)
@pytest.mark.parametrize("where", ["x", "dy"])
def test_infinities_reach_their_own_weights(ctx, dims, cin, cout, where):
    nx, ny, nz = dims
    V, B = nx * ny * nz, 2
    g = torch.Generator(device="cuda").manual_seed(cin + cout + nx)
    x = torch.randn((B, V, cin), generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn((B, V, cout), generator=g, device="cuda").to(torch.bfloat16).float()
    mag_x, mag_y = x.abs().double(), dy.abs().double()
    inf = float("inf")
    # the grid's last voxel, the end of a row inside it, and an inner one, in a channel each
    for q, (i, j, k) in enumerate([(nx - 1, ny - 1, nz - 1), (nx - 1, ny // 2, nz // 2), (nx // 2, ny // 2, 0)]):
        (x if where == "x" else dy)[1, i + nx * (j + ny * k), 3 * q + 1] = inf if q % 2 else -inf
    vol = lambda t: t.double().cpu().numpy().reshape(B, nz, ny, nx, -1)  # noqa: E731
    with np.errstate(invalid="ignore"):
        ref, rb = O.conv3d_backward_weights(vol(x), vol(dy))
    mag, mb = O.conv3d_backward_weights(vol(mag_x), vol(mag_y))
    assert np.isfinite(ref).any() and np.isinf(ref).any() and (where == "x") == (not np.isnan(ref).any())
    dw, db = _grads(ctx, dims, x, dy)
    _same(dw, ref, mag)
    _same(db, rb, mb)


@pytest.mark.parametrize("cin,cout", LAYERS)
def test_bias_sums_beyond_fp32_on_the_way(ctx, cin, cout):
    dims, B = (33, 18, 9), 2
    V = dims[0] * dims[1] * dims[2]
    x = torch.zeros((B, V, cin), dtype=torch.bfloat16, device="cuda")
    dy = torch.zeros((B, V, cout), device="cuda")
    dy[0, ::2], dy[1, 1::2] = 3e38, -3e38  # (each sample alone is beyond FP32's range)
    dy[1, 0] = 1.0
    if V % 2:
        dy[1, 2] = -3e38
    dy[:, 5, 0], dy[:, 5, 1] = float("inf"), float("-inf")
    dy[0, 7, 2], dy[1, 7, 2] = float("inf"), float("-inf")
    dy[1, 9, 3] = float("nan")
    ref = dy.double().sum((0, 1)).float()
    dw, db = _grads(ctx, dims, x, dy)
    assert np.isinf(db[:2]).all() and np.isnan(db[2:4]).all() and np.isfinite(db[4:]).all()
    assert np.array_equal(db[4:], ref[4:].double().cpu().numpy()) and db[0] > 0 > db[1]
