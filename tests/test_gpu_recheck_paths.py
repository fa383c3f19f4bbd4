"""The re-check counts, per pixel, the re-checked Gaussians that contribute
and stops after the last one while there are at most 256 of them; with more,
pixels are walked to their stop.  Both add the same float-pair terms of a
Gaussian, in FP64 and in any order, so a row re-checked among few equals the
row re-checked among all but for FP64 summation order (far below 1e-12)."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


def _solve(w, **kw):
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    s = flashsplat.Solver(w.gaussians, **kw)
    try:
        out = s.solve(w.cams, w.masks, w.E, w.gamma, table_dtype="float64")
        return {k: (v.cpu().numpy() if hasattr(v, "cpu") else v) for k, v in out.items()}
    finally:
        s.close()


@pytest.mark.parametrize("coverage,precision", [(0, 0), (1, 0), (0, 3)])
@pytest.mark.parametrize("size", [(113, 91), (16, 17)])
def test_few_rechecked_equal_all_rechecked(size, coverage, precision):
    w = synth.tiny_scene(n=3000, views=5, width=size[0], height=size[1], fx=1.2 * size[0])
    kw = {"coverage": coverage, "record_precision": precision}
    margin = _solve(w, recheck_margin=-1.0, **kw)["margin"]
    full = _solve(w, recheck_margin=1e30, **kw)
    order = np.argsort(margin)
    seen = int(np.isfinite(margin).sum())
    assert full["stats"].rechecked == seen
    for k in (1, 31, 33, 256, 257):
        if k >= seen:
            continue
        part = _solve(w, recheck_margin=float(np.nextafter(margin[order[k - 1]], np.float32(9))),
                      **kw)
        assert k <= part["stats"].rechecked < seen
        rows = order[:k]
        np.testing.assert_allclose(part["table"][rows], full["table"][rows], rtol=1e-12,
                                   atol=1e-15)
        assert np.array_equal(part["bits"][rows], full["bits"][rows])
