"""The workspace that bo_conv3d_backward_weights keeps with its context: the
partial sums of one thread block per SM and no more, none where the mma.sync
kernels run, and given back with the context."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_1606_00556_gb300 as bo  # noqa: E402

DIMS, B, C = (64, 16, 8), 2, 32
V = DIMS[0] * DIMS[1] * DIMS[2]
MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_one_partial_sum_per_sm_is_kept():
    bo.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    bo.bo_set_conv_engine(1)
    x = torch.randn(B, V, C, device="cuda").to(torch.bfloat16)
    room = torch.randn(B * V * C + 8, device="cuda")
    dw, db = torch.zeros(27, C, C, device="cuda"), torch.zeros(C, device="cuda")
    off = room[1:1 + B * V * C].view(B, V, C)  # (4 bytes off a 16-byte boundary: mma.sync)
    on = room[:B * V * C].view(B, V, C)
    warm = bo.Context(0)  # (modules and the allocator's own blocks)
    for dy in (off, on):
        bo.bo_conv3d_backward_weights(warm, DIMS, x, dy, dw, db)
    warm.close()
    ctx = bo.Context(0)
    start = _free()
    bo.bo_conv3d_backward_weights(ctx, DIMS, x, off, dw, db)
    assert start - _free() < MB
    bo.bo_conv3d_backward_weights(ctx, DIMS, x, on, dw, db)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    need = sms * (27 * C * C * 4 + C * 8 + 4)
    kept = start - _free()
    assert need <= kept <= need + 4 * MB  # (device memory comes in steps of 2 MB)
    for _ in range(3):
        bo.bo_conv3d_backward_weights(ctx, DIMS, x, on, dw, db)
    assert start - _free() == kept
    ctx.close()
    assert start - _free() < MB
