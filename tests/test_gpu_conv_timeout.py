"""Bounded waits of the tcgen05 convolutions: a launch with a wait that ran out
ends early, marks every output it did not reach as NaN and makes the calls
that synchronise return BO_ERR_TIMEOUT; the next call on the same context is
unaffected.

The wait is made to run out at a set tile of every block, the first or one
with copies and MMAs in flight before it; the block's other roles then end by
their own bounded waits, and nothing faults, traps or spins without a bound."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1606_00556_gb300 as bo  # noqa: E402

DIMS, B = (33, 18, 40), 4  # (several tiles a block)
V = DIMS[0] * DIMS[1] * DIMS[2]


@pytest.fixture
def ctx():
    bo.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    bo.bo_set_conv_engine(1)
    bo.bo_tc_status()
    yield bo.Context(0)
    bo.bo_set_conv_expire_tile(-1)
    bo.bo_tc_status()


def _expire(tile, fn):
    bo.bo_set_conv_expire_tile(tile)
    try:
        return fn()
    finally:
        bo.bo_set_conv_expire_tile(-1)


def _timeout(fn):
    with pytest.raises(bo.BoError) as e:
        fn()
    assert e.value.status == bo.BO_ERR_TIMEOUT


def _nan_or(got, want):
    keep = ~got.isnan()
    assert not keep.all() and torch.equal(got[keep], want[keep])


@pytest.mark.parametrize("tile", [0, 1, 3])
@pytest.mark.parametrize("cin,cout", [(16, 32), (32, 32), (32, 16)])
def test_single_layers_report_and_recover(ctx, tile, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(2)
    n = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    out = lambda *s, dtype=torch.float32: torch.full(s, 7.0, device="cuda", dtype=dtype)  # noqa: E731
    x, w, bias = n(B, V, cin).to(torch.bfloat16), n(27, cout, cin).to(torch.bfloat16), n(cout)
    dy = n(B, V, cout)
    dx, dw, db = out(B, V, cin), out(27, cout, cin), out(cout)

    def forward():
        y = out(B, V, cout, dtype=torch.bfloat16)
        yf = out(B, V, 4) if cout == 16 else None
        bo.bo_conv3d_forward(ctx, DIMS, x, w, bias, None, cout == 32, y, yf)
        torch.cuda.synchronize()
        return [y] if yf is None else [y, yf]

    def data():
        bo.bo_conv3d_backward_data(ctx, DIMS, dy.to(torch.bfloat16), w, dx)

    def weights():
        bo.bo_conv3d_backward_weights(ctx, DIMS, x, dy, dw, db)

    ref = forward()
    data()
    weights()
    good = [t.clone() for t in (dx, dw, db)]
    assert bo.bo_tc_status() == bo.BO_OK

    # a forward pass is asynchronous: the next call that synchronises reports it
    for got, want in zip(_expire(tile, forward), ref):
        _nan_or(got, want)
    assert bo.bo_tc_status() == bo.BO_ERR_TIMEOUT and bo.bo_tc_status() == bo.BO_OK
    _timeout(data)
    assert torch.equal(dx, good[0])
    _timeout(lambda: _expire(tile, data))
    _nan_or(dx, good[0])
    _timeout(lambda: _expire(tile, weights))
    assert dw.isnan().all() and db.isnan().all()
    # another context is not told of it
    bo.bo_set_conv_expire_tile(tile)
    bo.bo_conv3d_forward(ctx, DIMS, x, w, bias, None, cout == 32, out(B, V, cout, dtype=torch.bfloat16),
                         out(B, V, 4) if cout == 16 else None)
    torch.cuda.synchronize()
    bo.bo_set_conv_expire_tile(-1)
    bo.bo_conv3d_backward_data(bo.Context(0), DIMS, dy.to(torch.bfloat16), w, dx)
    _timeout(data)
    data()
    weights()
    assert all(torch.equal(a, b) for a, b in zip((dx, dw, db), good))


def test_network_backward_reports_and_recovers(ctx):
    net = bo.CNN(ctx, *DIMS, max_batch=B, seed=1)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((B, V, 16), generator=g, device="cuda").to(torch.bfloat16)
    target = torch.randn((B, V, 4), generator=g, device="cuda")
    loss = net.backward(x, target)
    grads = net.get_grads()
    assert np.isfinite(grads).all()
    _timeout(lambda: _expire(1, lambda: net.backward(x, target)))
    net.get_grads()  # (reported once)
    _expire(1, lambda: net.backward(x, target, want_loss=False))
    _timeout(net.get_grads)
    assert net.backward(x, target) == loss
    assert np.array_equal(net.get_grads(), grads)
    net.close()
