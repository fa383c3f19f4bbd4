"""Novel views whose tiles list 1 to 300 Gaussians: the render stages 128 at a
time and walks them in steps of four, two pixel rows per lane.  Against the
oracle at the bounds of the novel-view parity tests (1e-5 relative plus its
bound on near-threshold decisions), with faint Gaussians (no pixel stops) and
strong ones (pixels stop inside a step), in views that end inside a row pair."""
import numpy as np
import pytest

import oracle
from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opacity", [0.02, 0.7])
@pytest.mark.parametrize("n", [1, 4, 5, 127, 128, 129, 300])
def test_batches_of_records(n, opacity):
    import torch
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    rng = np.random.default_rng(n)
    g = {"mean": rng.uniform(-0.3, 0.3, (n, 3)).astype(np.float32),
         "quat": rng.standard_normal((n, 4)).astype(np.float32),
         "scale": rng.uniform(0.2, 0.6, (n, 3)).astype(np.float32),
         "opacity": (opacity * rng.uniform(0.9, 1.1, n)).astype(np.float32)}
    cams = [synth.camera((0.1, 0.2, -3.0), w, h, 20.0) for w, h in [(16, 16), (13, 5), (23, 12)]]
    bits = np.full(n, 2, np.uint64)
    s = flashsplat.Solver(g)
    try:
        r = s.render_masks(cams, torch.from_numpy(bits.astype(np.int64)).to(s.device), 2, tau=0.1,
                           want_planes=True)
        out = {k: [x.cpu().numpy() for x in r[k]] for k in ("masks", "rho", "depth")}
    finally:
        s.close()
    ora = oracle.render_masks(g, cams, bits, 2, tau=0.1)
    for v in range(len(cams)):
        ro, rr = ora.rho[v], ora.rho_risk[v]
        bound = 1e-5 * ro + 1.01 * rr + 1e-7
        assert np.all(np.abs(out["rho"][v] - ro) <= bound)
        seen = ro >= 1e-3
        dtol = 3e-5 * ora.depth[v] + (ora.z_risk[v] + ora.depth[v] * rr) / np.maximum(ro, 1e-30)
        assert np.all((np.abs(out["depth"][v] - ora.depth[v]) <= dtol + 1e-6)[seen])
        clear = np.abs(ro[0] - 0.1) > bound[0]
        assert np.array_equal(out["masks"][v][clear] == 1, (ro[0] > 0.1)[clear])
