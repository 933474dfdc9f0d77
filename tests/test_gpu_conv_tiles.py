"""The tcgen05 convolution kernels at the edges of their tiles: runs of 16,
32, 64 and 128 voxels with and without neighbours in another run, ragged rows
and columns, single planes and columns that several thread blocks share,
against the FP64 oracle with the bounds of the other convolution tests."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1606_00556_gb300 as bo  # noqa: E402
import test_gpu_cnn as T  # noqa: E402

DIMS = [(1, 1, 1), (2, 9, 3), (16, 8, 1), (17, 5, 4), (31, 7, 3), (33, 4, 5), (64, 3, 7), (65, 6, 2), (129, 2, 3),
        (200, 1, 2), (12, 12, 40)]


@pytest.fixture(scope="module")
def ctx():
    bo.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return bo.Context(0)


@pytest.fixture
def engine():
    bo.bo_set_conv_engine(1)
    yield
    assert bo.bo_tc_status() == bo.BO_OK  # no thread block gave up on a barrier


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("cin,cout,mode", T.COMBOS)
def test_forward(ctx, engine, dims, cin, cout, mode):
    T.test_conv_forward(ctx, dims, cin, cout, mode)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("cin,cout", [(16, 32), (32, 32), (32, 16)])
def test_gradients(ctx, engine, dims, cin, cout):
    T.test_conv_backward_data(ctx, dims, cin, cout)
    T.test_conv_backward_weights(ctx, dims, cin, cout)


@pytest.mark.parametrize("cin,cout", [(16, 32), (32, 32), (32, 16)])
def test_operands_on_16_byte_boundaries(ctx, engine, cin, cout):
    """Outputs off a 32-byte sector are stored in two halves: the same bits."""
    dims, B = (33, 5, 3), 2
    V = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cuda").manual_seed(5)

    def at(shape, off, dtype, fill=None):  # a tensor `off` bytes into its buffer
        n = 1
        for d in shape:
            n *= d
        k = off // (2 if dtype == torch.bfloat16 else 4)
        t = torch.empty(n + 64, device="cuda", dtype=dtype)[k:k + n].view(shape)
        return t if fill is None else t.copy_(fill)

    x = torch.randn((B, V, cin), generator=g, device="cuda").to(torch.bfloat16)
    w = torch.randn((27, cout, cin), generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn((B, V, cout), generator=g, device="cuda").to(torch.bfloat16)
    bias = torch.randn(cout, generator=g, device="cuda")
    outs = []
    for off in (0, 16):
        y = at((B, V, cout), off, torch.bfloat16)
        yf = at((B, V, 4), off, torch.float32) if cout == 16 else None
        dx = at((B, V, cin), off, torch.float32)
        bo.bo_conv3d_forward(ctx, dims, at(x.shape, off, x.dtype, x), at(w.shape, off, w.dtype, w), bias, None, cout == 32, y, yf)
        bo.bo_conv3d_backward_data(ctx, dims, at(dy.shape, off, dy.dtype, dy), at(w.shape, off, w.dtype, w), dx)
        torch.cuda.synchronize()
        outs.append([t.clone() for t in (y, yf, dx) if t is not None])
    assert all(torch.equal(a, b) for a, b in zip(*outs))
