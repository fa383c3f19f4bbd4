"""Every call whose kernels hold bounded waits reports a wait that ran out: the
removal's export and the mask render themselves, a solve and an accumulation at
fs_synchronize.  One wait is counted as run out by a test hook; nothing stalls."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


def test_a_wait_that_ran_out_is_reported():
    import torch
    from paper_2409_08270_gb300 import build, flashsplat as fsb
    build.build()
    w = synth.tiny_scene(n=500, views=2, width=48, height=40)
    s = fsb.Solver(w.gaussians)
    try:
        good = s.solve(w.cams, w.masks, w.E, w.gamma)
        table = torch.zeros((w.n, w.E), device="cuda")

        def accumulate():
            s.accumulate(w.cams, w.masks, w.E, table)
            fsb.fs_synchronize(s.ctx, torch.cuda.current_stream().cuda_stream)

        calls = [lambda: s.solve(w.cams, w.masks, w.E, w.gamma), accumulate,
                 lambda: s.keep_after_removal(good["bits"], [1]),
                 lambda: s.render_masks(w.cams, good["bits"], w.E)]
        fsb.fs_test_wait_timeout(s.ctx, True)
        for call in calls:
            with pytest.raises(fsb.FlashSplatError) as ei:
                call()
            assert ei.value.status == fsb.FS_TIMEOUT
        fsb.fs_test_wait_timeout(s.ctx, False)
        for call in calls:
            call()
        assert np.array_equal(s.solve(w.cams, w.masks, w.E, w.gamma)["bits"].cpu().numpy(),
                              good["bits"].cpu().numpy())
    finally:
        s.close()


def test_a_render_keeps_an_unfinished_solves_counters():
    """The render counts in words of its own: a solve still in flight reports
    its out-of-range labels afterwards."""
    import torch
    from paper_2409_08270_gb300 import build, flashsplat as fsb
    build.build()
    w = synth.tiny_scene(n=500, views=2, width=48, height=40)
    masks = [np.where(np.arange(m.size).reshape(m.shape) < 7, 200, m).astype(np.uint8)
             for m in w.masks]
    s = fsb.Solver(w.gaussians)
    try:
        r = s.solve(w.cams, masks, w.E, w.gamma, sync=False)
        s.render_masks(w.cams, r["bits"], w.E)
        st = fsb.fs_synchronize(s.ctx, torch.cuda.current_stream().cuda_stream)
        assert st.bad_labels == 14
    finally:
        s.close()


def test_the_wait_limit_is_seconds():
    """The limit on the polls of a look-back wait amounts to some two seconds,
    by the time a sixteenth of them takes (at most a quarter of a second)."""
    import os
    import re
    import time
    from paper_2409_08270_gb300 import build, flashsplat as fsb
    build.build()
    text = open(os.path.join(build.CSRC, "fs_internal.h")).read()
    polls = 1 << int(re.search(r"kLookbackSpinLimit = 1 << (\d+)", text).group(1))
    assert fsb.fs_check_wait_timeout(0, 1) == fsb.FS_TIMEOUT
    t = time.perf_counter()
    assert fsb.fs_check_wait_timeout(0, polls // 16) == fsb.FS_TIMEOUT
    assert time.perf_counter() - t < 0.25
