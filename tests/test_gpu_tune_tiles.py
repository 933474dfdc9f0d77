"""The batch autotuner tries tiles of the per-kernel AMG form only where a
realisation launches it: systems whose levels all run in one thread-block
cluster are the same graph under every tile, and keep the default one."""
import pytest

import bogen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,tiled", [([(20, 20, 5), (16, 10, 4), (40, 36, 10)], False),
                                        ([(20, 20, 5), (62, 45, 19)], True)])
def test_tiles_are_tried_where_they_are_launched(dims, tiled, tmp_path):
    import paper_1606_00556_gb300 as bo
    bo.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    ctx = bo.Context(0)
    mats, precs, bs = [], [], []
    for q, d in enumerate(dims):
        a = bogen.assemble(bogen.ensemble_case(dict(dims=d, sigma=1.0, seed=q)))
        mats.append(bo.Matrix.from_bsr(ctx, bo.grid(*d), a["rowptr"], a["col"], a["val"]))
        precs.append(bo.Preconditioner(mats[-1]))
        bs.append(torch.tensor(a["b"], dtype=torch.float64, device="cuda"))
    r = bo.bo_autotune_batched(precs, bs, [torch.zeros_like(b) for b in bs], cache_path=str(tmp_path / "t.json"))
    bo.bo_set_batch_streams(16)
    if r["launch_mode"] == bo.BO_LAUNCH_STREAM:
        assert not any(r["tile_ms"])
    elif tiled:
        assert len(set(r["tile_ms"])) > 1
    else:
        assert r["tile_ms"] == [r["best_ms"]] * 5 and r["best_ms"] == min(r["trial_ms"])
        assert (r["amg_cells"], r["amg_threads"]) == (1, 256)
