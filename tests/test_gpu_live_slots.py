"""Large depth chunks are reduced to their live slots before the binning
(chunks of 2^22 positions and more, with a fifth of the batch's slots).  One
chunk never is, so six chunks must give the table of one: the same FP32 terms
summed in FP64 in another order, far below 1e-12 relative.  The views hold one
whose prefix table is too large for shared memory and ragged ones; the
Gaussian count leaves a partial word of slot bits."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


def _workload():
    rng = np.random.default_rng(7)
    n = 260_003
    sizes = [(2600, 1030)] + [(int(rng.integers(17, 200)), int(rng.integers(17, 160)))
                              for _ in range(46)]
    gauss = {"mean": rng.uniform(-1, 1, (n, 3)).astype(np.float32),
             "quat": rng.standard_normal((n, 4)).astype(np.float32),
             "scale": np.exp(rng.normal(-4, 1, (n, 3))).astype(np.float32),
             "opacity": (1 / (1 + np.exp(-rng.normal(0, 1.5, n)))).astype(np.float32)}
    cams, masks = [], []
    for k, (w, h) in enumerate(sizes):
        az = 0.13 * k
        cams.append(synth.camera((3 * np.sin(az), 0.3, -3 * np.cos(az)), w, h, 1.1 * w))
        m = rng.integers(0, 3, (h, w)).astype(np.uint8)
        m[: h // 3] = 9  # out of range: tiles that start saturated
        masks.append(m)
    return gauss, cams, masks


@pytest.mark.parametrize("coverage", [0, 1])
def test_live_slots_change_no_result(coverage):
    import torch
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    gauss, cams, masks = _workload()
    out = {}
    for chunks in (1, 6):
        s = flashsplat.Solver(gauss, depth_chunks=chunks, views_per_batch=47, coverage=coverage)
        try:
            dm = s.upload_masks(masks)
            r = s.solve(cams, dm, 3, 0.3, table_dtype="float64")
            out[chunks] = (r["table"].cpu().numpy(), r["bits"].cpu().numpy())
            if chunks == 6:
                g = s.capture(cams, dm, 3, 0.3, table_dtype="float64")
                g.launch()
                g.synchronize()
                torch.cuda.synchronize()
                out["graph"] = (g.outputs["table"].cpu().numpy(), g.outputs["bits"].cpu().numpy())
                g.close()
        finally:
            s.close()
    assert (out[1][0] > 0).any()
    for key in (6, "graph"):
        np.testing.assert_allclose(out[key][0], out[1][0], rtol=1e-12, atol=1e-14)
        assert np.array_equal(out[key][1], out[1][1])
