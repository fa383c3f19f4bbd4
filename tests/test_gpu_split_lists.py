"""Lists that are too long, or for which there is no memory, are made in parts.
The main pass cuts a depth chunk of its own choosing by positions, and keeps
every part's list for the re-check; the re-check's own binning goes by views.
All must give what six explicit chunks give: the same FP32 terms summed in FP64
in another order, far below 1e-12 relative, and the same decisions."""
import numpy as np
import pytest

from paper_2409_08270_gb300 import synth

pytestmark = pytest.mark.gpu


def _workload(n, side, scale):
    rng = np.random.default_rng(3)
    V = 50
    g = {"mean": rng.uniform(-1, 1, (n, 3)).astype(np.float32),
         "quat": rng.standard_normal((n, 4)).astype(np.float32),
         "scale": np.full((n, 3), scale, np.float32),
         "opacity": rng.uniform(0.01, 0.03, n).astype(np.float32)}
    cams = [synth.camera((3 * np.sin(0.1 * k), 0, -3 * np.cos(0.1 * k)), side, side, 1.1 * side)
            for k in range(V)]
    return g, cams, [rng.integers(0, 2, (side, side)).astype(np.uint8) for _ in range(V)]


def _solve(g, cams, masks, **kw):
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    s = flashsplat.Solver(g, **kw)
    try:
        r = s.solve(cams, masks, 2, 0.0, table_dtype="float64")
        return r["table"].cpu().numpy(), r["bits"].cpu().numpy(), r["stats"]
    finally:
        s.close()


def _same(a, b):
    np.testing.assert_allclose(a[0], b[0], rtol=1e-12, atol=1e-14)
    assert np.array_equal(a[1], b[1])


def test_more_entries_than_one_list_holds():
    """More than 2^31 entries over all depths, 2^29 at most in a part."""
    from paper_2409_08270_gb300 import flashsplat
    work = _workload(250_000, 512, 0.42)
    kw = {"recheck_margin": 1e-4}
    with pytest.raises(flashsplat.FlashSplatError) as ei:
        _solve(*work, depth_chunks=1, **kw)
    assert ei.value.status == flashsplat.FS_UNSUPPORTED
    six = _solve(*work, depth_chunks=6, **kw)
    own = _solve(*work, **kw)                             # kept parts
    assert own[2].rechecked > 0 and own[2].recheck_rebinned == 0
    _same(own, six)
    _same(_solve(*work, recheck_reproject=True, **kw), six)  # the re-check bins by views


def test_captured_solve_fits_where_six_chunks_do():
    """A capture's plan cannot cut its chunks: it takes more of them instead."""
    import torch
    from paper_2409_08270_gb300 import flashsplat
    g, cams, masks = _workload(125_000, 256, 0.38)
    six = _solve(g, cams, masks, depth_chunks=6, recheck_margin=1e-4)

    def captured(chunks, held_to=None):
        s = flashsplat.Solver(g, depth_chunks=chunks, recheck_margin=1e-4)
        held = graph = None
        try:
            dm = s.upload_masks(masks)
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            if held_to:
                held = torch.empty(free - held_to, dtype=torch.uint8, device="cuda")
            graph = s.capture(cams, dm, 2, 0.0, table_dtype="float64")
            used = free - torch.cuda.mem_get_info()[0]
            graph.launch()
            graph.synchronize()
            out = graph.outputs
            return used, (out["table"].cpu().numpy(), out["bits"].cpu().numpy())
        finally:
            if graph is not None:
                graph.close()
            s.close()
            del held
            torch.cuda.empty_cache()

    used, first = captured(6)
    _same(first, six)
    _same(captured(0, used + used // 5)[1], six)


def test_lists_that_do_not_fit_in_memory():
    """With no more memory than six chunks take and a fifth."""
    import torch
    g, cams, masks = work = _workload(125_000, 256, 0.38)
    kw = {"recheck_margin": 1e-4}
    _solve(*work, depth_chunks=6, **kw)                  # kernels loaded, masks' memory cached
    from paper_2409_08270_gb300 import flashsplat
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s = flashsplat.Solver(g, depth_chunks=6, **kw)
    try:
        s.solve(cams, masks, 2, 0.0, table_dtype="float64")
        used = free - torch.cuda.mem_get_info()[0]
    finally:
        s.close()
    torch.cuda.synchronize()
    six = _solve(*work, depth_chunks=6, **kw)
    held = torch.empty(torch.cuda.mem_get_info()[0] - used - used // 5, dtype=torch.uint8,
                       device="cuda")
    try:
        with pytest.raises(flashsplat.FlashSplatError) as ei:
            _solve(*work, depth_chunks=1, **kw)
        assert ei.value.status == flashsplat.FS_OUT_OF_MEMORY
        own = _solve(*work, **kw)
    finally:
        del held
        torch.cuda.empty_cache()
    _same(own, six)
