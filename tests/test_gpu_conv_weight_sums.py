"""The sums of the tcgen05 weight gradient: dY is rounded to BF16 for the
products but summed unrounded for the bias, and the bias sum keeps as much as
an FP64 sum."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1606_00556_gb300 as bo  # noqa: E402
from oracle import cnn as O  # noqa: E402

LAYERS = [(16, 32), (32, 32), (32, 16)]
DIMS = [(17, 5, 4), (33, 18, 9)]


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
    return dw, db


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("cin,cout", LAYERS)
def test_products_take_rounded_values_and_the_bias_unrounded_ones(ctx, dims, cin, cout):
    V, B = dims[0] * dims[1] * dims[2], 2
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    x = torch.randn((B, V, cin), generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn((B, V, cout), generator=g, device="cuda")
    dw, db = _grads(ctx, dims, x, dy)
    vol = lambda t: t.double().cpu().numpy().reshape(B, dims[2], dims[1], dims[0], -1)  # noqa: E731
    X, D = vol(x), vol(dy.to(torch.bfloat16))
    ref, _ = O.conv3d_backward_weights(X, D)
    mag, _ = O.conv3d_backward_weights(np.abs(X), np.abs(D))
    assert (np.abs(dw.double().cpu().numpy() - ref) <= 1e-5 * mag + 1e-30).all()  # (FP32 accumulation)
    d = dy.cpu().numpy().reshape(-1, cout)
    for c in range(cout):
        exact = math.fsum(d[:, c].tolist())
        # the sum itself to well below FP32, one rounding of the result
        assert abs(float(db[c]) - exact) <= 2.0 ** -24 * abs(exact) + 2.0 ** -50 * float(np.abs(d[:, c].astype(np.float64)).sum())


@pytest.mark.parametrize("cin,cout", LAYERS)
def test_the_bias_sum_cancels_as_in_fp64(ctx, cin, cout):
    """Values of which every FP64 sum is exact (multiples of 2^-30, sum of magnitudes below 2^23): a few
    large ones that cancel, and small ones that do but for a few units."""
    dims, B = (33, 18, 9), 2
    BV = dims[0] * dims[1] * dims[2] * B
    rng = np.random.default_rng(cin * cout)
    d = np.zeros((BV, cout))
    for c in range(cout):
        half = rng.integers(2 ** 23, 2 ** 24, (BV - 9) // 2)  # (24 bits, so that two of them take 25)
        small = np.concatenate([half, -half, np.zeros((BV - 9) % 2, np.int64)])
        v = np.concatenate([[2.0 ** 49, -2.0 ** 49] * 4, [c + 1.0], small])
        v = v[rng.permutation(BV)] * 2.0 ** -30
        d[:, c] = v
    assert np.array_equal(d, d.astype(np.float32).astype(np.float64))
    sums = [math.fsum(d[:, c].tolist()) for c in range(cout)]
    assert sums == [(c + 1) * 2.0 ** -30 for c in range(cout)] and np.abs(d).sum(0).max() < 2.0 ** 23
    dy = torch.from_numpy(d.astype(np.float32)).view(B, -1, cout).cuda()
    x = torch.zeros((B, BV // B, cin), dtype=torch.bfloat16, device="cuda")
    dw, db = _grads(ctx, dims, x, dy)
    assert db.double().cpu().tolist() == [float(np.float32(s)) for s in sums]
    assert not dw.any()
