"""A request is admitted by an estimate of the device memory it needs, which
must not lie below what a scene of few entries a slot then takes: the window of
a full batch, and, with the one depth chunk that small scenes take, the lists
of all its views."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views,size", [(100_000, 12, (512, 512)), (60_000, 24, (320, 240)),
                                          (400_000, 8, (1008, 756))])
def test_estimate_covers_what_is_taken(n, views, size):
    import torch
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    rng = np.random.default_rng(n)
    g = {"mean": rng.uniform(-1, 1, (n, 3)).astype(np.float32),
         "quat": rng.standard_normal((n, 4)).astype(np.float32),
         "scale": np.exp(rng.normal(-4, 1, (n, 3))).astype(np.float32),
         "opacity": rng.uniform(0.05, 0.9, n).astype(np.float32)}
    cams = [synth.camera((4 * np.sin(0.1 * k), 0, -4 * np.cos(0.1 * k)), *size, 1.1 * size[0])
            for k in range(views)]
    masks = [(rng.random(size[::-1]) < 0.3).astype(np.uint8) for _ in cams]
    tiny = synth.tiny_scene(n=500, views=2, width=48, height=40)
    srv = flashsplat.Server(slots=1)
    try:
        small, sid = srv.add_scene(tiny.gaussians), srv.add_scene(g)
        srv.fetch(srv.submit(small, tiny.cams, tiny.masks, tiny.E, 0.0))   # kernels loaded
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        info = srv.fetch(srv.submit(sid, cams, masks, 2, 0.0))["info"]
        used = free - torch.cuda.mem_get_info()[0]
    finally:
        srv.close()
    assert used <= info.bytes_estimate
