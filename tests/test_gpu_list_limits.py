"""What binning does where lists get long.

* A solve that chooses its own number of depth chunks halves a chunk of more
  than 2^29 list entries; the table must be that of six explicit chunks (the
  same FP32 terms summed in FP64 in another order: far below 1e-12 relative),
  and so must the re-check's decisions, which then bins anew.
* The allocation-free solve bins a view at once where its entries fit, and in
  six chunks where they do not.  Its FP32 table meets the FP64 one within the
  rounding of its atomic additions: at most one per 8x8 sub-tile of the view
  and Gaussian, 4096 of 2^-24 relative each."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


def _fsb():
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    return flashsplat


def test_a_chunk_with_too_many_entries_is_halved():
    fsb = _fsb()
    rng = np.random.default_rng(3)
    n, V, side = 250_000, 50, 256
    g = {"mean": rng.uniform(-1, 1, (n, 3)).astype(np.float32),
         "quat": rng.standard_normal((n, 4)).astype(np.float32),
         "scale": np.full((n, 3), 0.38, np.float32),
         "opacity": rng.uniform(0.01, 0.03, n).astype(np.float32)}
    cams = [synth.camera((3 * np.sin(0.1 * k), 0, -3 * np.cos(0.1 * k)), side, side, 281.0)
            for k in range(V)]
    masks = [rng.integers(0, 2, (side, side)).astype(np.uint8) for _ in range(V)]
    out = {}
    for chunks in (1, 0, 6):
        s = fsb.Solver(g, depth_chunks=chunks, recheck_margin=1e-3)
        try:
            r = s.solve(cams, masks, 2, 0.0, table_dtype="float64")
            out[chunks] = (r["table"].cpu().numpy(), r["bits"].cpu().numpy(), r["stats"])
        finally:
            s.close()
    assert out[1][2].list_entries > 1 << 29 > out[0][2].list_entries
    assert out[0][2].rechecked > 0
    for chunks in (1, 6):
        np.testing.assert_allclose(out[0][0], out[chunks][0], rtol=1e-12, atol=1e-14)
        assert np.array_equal(out[0][1], out[chunks][1])


@pytest.mark.parametrize("scale", [0.02, 0.15])
def test_noalloc_one_list_or_six(scale):
    import torch
    fsb = _fsb()
    w = synth.tiny_scene(n=16_384, views=1, width=512, height=512, fx=440.0)
    rng = np.random.default_rng(4)
    gauss = dict(w.gaussians)
    gauss["scale"] = np.full((w.n, 3), scale, np.float32)
    gauss["opacity"] = rng.uniform(0.3, 0.95, w.n).astype(np.float32)
    s = fsb.Solver(gauss, recheck_margin=-1.0, depth_chunks=1)
    try:
        r = s.solve(w.cams, w.masks, w.E, w.gamma, table_dtype="float64")
        want, entries = r["table"].cpu().numpy(), r["stats"].list_entries
    finally:
        s.close()
    assert (entries > 1 << 19) == (scale > 0.1)      # both ways are taken
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in gauss.items()}
    g = fsb.fs_gaussians(n=w.n, mean=dev["mean"].data_ptr(), quat=dev["quat"].data_ptr(),
                         scale=dev["scale"].data_ptr(), opacity=dev["opacity"].data_ptr(),
                         quat_dtype=fsb.FS_F32, scale_dtype=fsb.FS_F32, opacity_dtype=fsb.FS_F32,
                         memory=fsb.FS_MEM_DEVICE)
    masks = [torch.from_numpy(m).cuda() for m in w.masks]
    table = torch.empty((w.n, w.E), device="cuda")
    fsb.fs_solve_noalloc(0, g, fsb.make_cameras(w.cams), [m.data_ptr() for m in masks], fsb.FS_U8,
                         w.E, w.gamma, table.data_ptr())
    torch.cuda.synchronize()
    np.testing.assert_allclose(table.cpu().numpy(), want, rtol=4096 * 2.0 ** -24, atol=1e-7)
