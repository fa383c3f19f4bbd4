"""After a bounded wait has given up, words of its launch's outputs are missing;
what follows must not index memory by them.  With one wait counted as run out
from the start (a test hook; nothing stalls), sorts, compactions, binnings and
tile ranges do nothing, the call itself returns FS_TIMEOUT at the next count it
reads back, and the caller's table stays as it was."""
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("table_dtype", ["float32", "float64"])
def test_nothing_is_listed_after_a_wait_gave_up(table_dtype):
    import torch
    from paper_2409_08270_gb300 import build, flashsplat as fsb
    build.build()
    w = synth.tiny_scene(n=3000, views=3, width=113, height=91)
    s = fsb.Solver(w.gaussians)
    try:
        table = torch.zeros((w.n, w.E), device="cuda", dtype=getattr(torch, table_dtype))
        fsb.fs_test_wait_timeout(s.ctx, True)
        with pytest.raises(fsb.FlashSplatError) as ei:
            s.accumulate(w.cams, w.masks, w.E, table)
        assert ei.value.status == fsb.FS_TIMEOUT
        with pytest.raises(fsb.FlashSplatError) as ei:
            s.solve(w.cams, w.masks, w.E, w.gamma, sync=False)
        assert ei.value.status == fsb.FS_TIMEOUT
        torch.cuda.synchronize()
        assert not table.any()
        fsb.fs_test_wait_timeout(s.ctx, False)
        s.accumulate(w.cams, w.masks, w.E, table)
        torch.cuda.synchronize()
        assert table.any()
    finally:
        s.close()
