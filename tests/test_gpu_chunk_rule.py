"""The number of depth chunks a solve chooses follows its Gaussians, its views'
tiles and its number of views, not the Gaussians alone: 300,000 Gaussians in
thirty 1600x1200 views take several chunks (one was 12 % slower than six), in
one such view, or in small ones, a single chunk.  A served request reports it."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,size,views,least,most", [
    (300_000, (1600, 1200), 30, 2, 4),
    (300_000, (1600, 1200), 1, 1, 1),
    (300_000, (160, 120), 40, 1, 1),
    (2_000, (128, 128), 8, 1, 1)])
def test_chunks_chosen(n, size, views, least, most):
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    rng = np.random.default_rng(n + views)
    g = {"mean": rng.uniform(-1, 1, (n, 3)).astype(np.float32),
         "quat": rng.standard_normal((n, 4)).astype(np.float32),
         "scale": np.full((n, 3), 0.01, np.float32),
         "opacity": rng.uniform(0.2, 0.9, n).astype(np.float32)}
    cams = [synth.camera((4 * np.sin(0.02 * k), 0, -4 * np.cos(0.02 * k)), *size, 1.1 * size[0])
            for k in range(views)]
    mask = np.zeros(size[::-1], np.uint8)
    srv = flashsplat.Server(slots=1)
    try:
        sid = srv.add_scene(g)
        info = srv.fetch(srv.submit(sid, cams, [mask] * views, 2, 0.0))["info"]
    finally:
        srv.close()
    assert least <= info.depth_chunks <= most
