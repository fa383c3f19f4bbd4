"""The server's tuner offers the chunks that an untuned request takes: a scene of
100,000 Gaussians in small views takes one by its size (solved 1.3 times as fast
as with four), so tuning ends at one, two or three, with unchanged results."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


def test_tuned_chunks_follow_the_size():
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    w = synth.binary_scene(n=100_000, views=8, width=300, height=200)
    plain, tuned = flashsplat.Server(slots=1), flashsplat.Server(slots=1, autotune=True)
    try:
        a = plain.fetch(plain.submit(plain.add_scene(w.gaussians), w.cams, w.masks, w.E, 0.5))
        sid = tuned.add_scene(w.gaussians)
        b = [tuned.fetch(tuned.submit(sid, w.cams, w.masks, w.E, 0.5)) for _ in range(2)]
    finally:
        plain.close()
        tuned.close()
    assert a["info"].depth_chunks == 1
    for r in b:
        assert r["info"].depth_chunks <= 3
        decided = (a["margin"] > 1e-9) & (r["margin"] > 1e-9)
        assert np.array_equal(a["label"][decided], r["label"][decided])
