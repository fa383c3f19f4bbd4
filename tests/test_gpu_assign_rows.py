"""The FP64 assignment has a short form for rows of contributions and the
general one for the rest (negative or non-finite entries, sums at the clamp of
the normalisation or near overflow).  Both against Listing 1's comparison in
numpy: decisions equal wherever the two sides differ by more than 1e-12 of the
row's normalisation (each side's rounding is a few 2^-53), and exactly on rows
of small integers, where no step rounds; margins to 1e-6 (FP32 outputs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _general(t, gamma):
    g = float(np.float32(gamma))
    with np.errstate(all="ignore"):
        S = t.sum(1, keepdims=True)
        others = S - t
        nrm = np.maximum(np.abs(others) + np.abs(t), 1e-12)
        lhs, rhs = t - others, g * nrm
        margin = np.where(S > 0, np.abs((1 - g) * t - (1 + g) * others) / S, np.inf).min(1)
    return lhs, rhs, nrm, margin, S[:, 0]


@pytest.mark.parametrize("E", [1, 2, 4, 5, 33, 64])
@pytest.mark.parametrize("gamma", [-1.0, -0.4, 0.0, 0.5, 1.0])
def test_fp64_rows(E, gamma):
    import torch
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    rng = np.random.default_rng(E)
    n = 4099
    t = rng.random((n, E)) ** 4 * np.exp(rng.normal(0, 6, (n, 1)))
    t[:1000] = rng.integers(0, 5, (1000, E))          # exact ties, empty rows
    t[1000:1100] *= -1.0
    t[1100:1200, 0] = -0.0
    t[1200:1300] = rng.random((100, E)) * 1e-13       # below the normalisation's clamp
    t[1300:1310] = 1e305
    s = flashsplat.Solver({"mean": np.zeros((1, 3), np.float32),
                           "quat": np.ones((1, 4), np.float32),
                           "scale": np.ones((1, 3), np.float32),
                           "opacity": np.ones(1, np.float32)})
    try:
        bits, label, margin = s.assign(torch.from_numpy(t).cuda(), gamma)
        bits, label, margin = bits.cpu().numpy(), label.cpu().numpy(), margin.cpu().numpy()
    finally:
        s.close()
    lhs, rhs, nrm, want_margin, S = _general(t, gamma)
    member = lhs > rhs
    got = (bits.view(np.uint64)[:, None] >> np.arange(E, dtype=np.uint64)) & np.uint64(1) == 1
    clear = np.abs(lhs - rhs) > 1e-12 * nrm
    clear[:1000] = True if gamma in (-1.0, 0.0, 0.5, 1.0) else clear[:1000]
    assert np.array_equal(got[clear], member[clear])
    one = got.sum(1) == 1
    assert np.array_equal(label, np.where(one, got.argmax(1), -1))
    fin = np.isfinite(want_margin) & (S > 0)
    np.testing.assert_allclose(margin[fin], want_margin[fin], rtol=1e-6, atol=1e-12)


@pytest.mark.parametrize("E", [5, 8, 33, 95])
@pytest.mark.parametrize("skip", [0, 1, 3])
def test_rows_at_any_alignment(E, skip):
    """The staged form copies 16 bytes at a time from 16-byte boundaries; tables
    that start elsewhere, and the last partial block, give the same decisions
    as an aligned copy, exactly."""
    import torch
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(E)
    for dtype in (torch.float32, torch.float64):
        full = torch.rand((1000 + skip, E), generator=g, device="cuda", dtype=dtype)
        s = flashsplat.Solver({"mean": np.zeros((1, 3), np.float32),
                               "quat": np.ones((1, 4), np.float32),
                               "scale": np.ones((1, 3), np.float32),
                               "opacity": np.ones(1, np.float32)})
        try:
            a = s.assign(full[skip:], 0.1)
            b = s.assign(full[skip:].clone(), 0.1)
            for x, y in zip(a, b):
                assert (x is None and y is None) or torch.equal(x, y)
        finally:
            s.close()
