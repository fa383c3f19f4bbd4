"""Above 256 re-checked Gaussians the re-check finds them in the tiles' lists
and a pixel's walk still ends at its last one.  Rows equal those re-checked
among all but for FP64 summation order (far below 1e-12)."""
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


@pytest.mark.parametrize("coverage,precision,chunks", [(0, 0, 0), (0, 0, 6), (1, 0, 3), (0, 3, 0)])
def test_one_more_rechecked_is_no_longer_walk(coverage, precision, chunks):
    """Faint Gaussians, of which few are re-checked at any pixel: above 256 of
    them the last one still ends a pixel's walk, so that one more costs about
    its share of pairs and not every pixel's whole list."""
    w = synth.tiny_scene(n=40_000, views=5, width=113, height=91, fx=135.0)
    rng = np.random.default_rng(5)
    w.gaussians["opacity"] = rng.uniform(0.01, 0.03, w.n).astype(np.float32)
    w.gaussians["scale"] = np.full((w.n, 3), 0.02, np.float32)
    kw = {"coverage": coverage, "record_precision": precision, "depth_chunks": chunks}
    margin = _solve(w, recheck_margin=-1.0, **kw)["margin"]
    full = _solve(w, recheck_margin=1e30, **kw)
    order = np.argsort(margin)
    runs = {}
    for k in (256, 257, 300):
        runs[k] = _solve(w, recheck_margin=float(np.nextafter(margin[order[k - 1]], np.float32(9))),
                         **kw)
        assert k <= runs[k]["stats"].rechecked <= k + 3
        rows = order[:k]
        np.testing.assert_allclose(runs[k]["table"][rows], full["table"][rows], rtol=1e-12,
                                   atol=1e-15)
        assert np.array_equal(runs[k]["bits"][rows], full["bits"][rows])
    pairs = {k: r["stats"].recheck_pairs for k, r in runs.items()}
    assert pairs[300] < 1.3 * pairs[256]
