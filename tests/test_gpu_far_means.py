"""Thin Gaussians whose means project some 10^6 pixels outside the image
still cross it.  Moving the principal point by (4, 2) pixels moves every pixel
by as much and leaves all its alphas; the re-check's float pairs see that to
better than 1e-8, so its rows may differ by no more than 1e-6 -- whatever
pieces of tiles the pixels fall into then."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FX, SIDE = 500.0, 96


def _scene():
    rng = np.random.default_rng(11)
    n = 200
    z = rng.uniform(0.25, 0.4, n)
    theta = rng.uniform(0.15, 1.4, n) * rng.choice([-1, 1], n)
    far = rng.uniform(3e5, 1.2e6, n)
    px = 48 - far * np.cos(theta) + rng.uniform(-20, 20, n)   # the long axis crosses the image
    py = 48 - far * np.sin(theta) + rng.uniform(-20, 20, n)
    mean = np.stack([(px - 48) * z / FX, (py - 48) * z / FX, z], 1)
    quat = np.stack([np.cos(theta / 2), 0 * z, 0 * z, np.sin(theta / 2)], 1)
    scale = np.stack([0.6 * far * z / FX, 1e-5 + 0 * z, 1e-5 + 0 * z], 1)
    return {"mean": mean.astype(np.float32), "quat": quat.astype(np.float32),
            "scale": scale.astype(np.float32),
            "opacity": rng.uniform(0.02, 0.2, n).astype(np.float32)}


def _camera(dx, dy):
    return {"R": np.eye(3), "t": np.zeros(3), "fx": FX, "fy": FX, "cx": 48.0 + dx,
            "cy": 48.0 + dy, "width": SIDE + 16, "height": SIDE + 16}


def _rows(dx, dy, **kw):
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    label = np.random.default_rng(2).integers(0, 2, (SIDE, SIDE)).astype(np.uint8)
    mask = np.full((SIDE + 16, SIDE + 16), 9, np.uint8)       # 9: no label
    mask[dy:dy + SIDE, dx:dx + SIDE] = label
    s = flashsplat.Solver(_scene(), recheck_margin=1e30, **kw)
    try:
        r = s.solve([_camera(dx, dy)], [mask], 2, 0.0, table_dtype="float64")
        return r["table"].cpu().numpy(), r["stats"].rechecked
    finally:
        s.close()


@pytest.mark.parametrize("reproject", [False, True])
def test_rows_do_not_depend_on_the_pieces(reproject):
    a, seen = _rows(0, 0, recheck_reproject=reproject)
    assert seen > 100
    for dx, dy in ((4, 2), (3, 1), (9, 5)):
        b, _ = _rows(dx, dy, recheck_reproject=reproject)
        np.testing.assert_allclose(b, a, rtol=1e-6, atol=1e-9)
