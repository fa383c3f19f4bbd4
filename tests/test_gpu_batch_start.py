"""The state at the start of a batch (pixels with and without a label, tiles
and sub-tiles that begin saturated) is written by warps that take two
sub-tiles and blocks that take four tiles: views of one to nine tiles, ragged
and mixed in one batch, with whole sub-tiles, whole tiles and single pixels
out of range, against the oracle at the parity tests' tolerance, and the
count of bad labels exactly."""
import numpy as np
import pytest

import oracle
from paper_2409_08270_gb300 import synth
from parity import label_check, table_errors

pytestmark = pytest.mark.gpu

SIZES = [(16, 16), (17, 9), (40, 33), (64, 16), (71, 15), (8, 70), (1, 1), (48, 48)]


@pytest.mark.parametrize("dtype", [np.uint8, np.int32])
@pytest.mark.parametrize("batch", [1, 3, 0])
def test_batch_start(dtype, batch):
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    rng = np.random.default_rng(11)
    gauss = synth.tiny_scene(n=700, views=1, width=16, height=16).gaussians
    cams, masks = [], []
    for k, (w, h) in enumerate(SIZES):
        cams.append(synth.camera((3 * np.sin(k), 0.2, -3 * np.cos(k)), w, h, 1.2 * max(w, h)))
        m = rng.integers(0, 3, (h, w)).astype(dtype)
        for y in range(0, h, 8):
            for x in range(0, w, 8):
                if rng.random() < 0.3:
                    m[y:y + 8, x:x + 8] = 200
        if k % 3 == 2:
            m[16:32, :16] = 3
        m[rng.random((h, w)) < 0.05] = 77 if dtype == np.uint8 else -5
        masks.append(m)
    s = flashsplat.Solver(gauss, views_per_batch=batch)
    try:
        r = s.solve(cams, masks, 3, 0.2, table_dtype="float64")
        table, bits = r["table"].cpu().numpy(), r["bits"].cpu().numpy()
        bad = r["stats"].bad_labels
    finally:
        s.close()
    acc = oracle.accumulate(gauss, cams, masks, 3)
    assert bad == acc.n_bad_label == sum(int(((m < 0) | (m >= 3)).sum()) for m in masks) > 0
    assert table_errors(table, acc.table, acc.risk, rtol=1e-5)[2]["violations"] == 0
    lab = label_check(bits, acc.table, acc.risk, 0.2, table_rtol=1e-5)
    assert lab["mismatch_outside_window"] == 0
