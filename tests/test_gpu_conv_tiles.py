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
