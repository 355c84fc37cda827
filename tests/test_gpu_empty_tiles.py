"""Tiles that no Gaussian reaches, in the walks by 8-lane groups: they read their targets (a value that is not
finite still fails the call), write zeros where an image or a gradient is asked for, and cost little besides
that. A large image of a small object, or the sky of an outdoor one, is mostly such tiles."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
W, H = 1600, 1060


@pytest.fixture(scope="module")
def icgs():
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs as I
    I.load()
    return I


def _one_gaussian(icgs, cams, w, h):
    import numpy as np
    sc = icgs.Scene(torch.zeros((1, 3), device=DEV), torch.full((1, 3), 0.02, device=DEV),
                    torch.tensor([[1.0, 0.0, 0.0, 0.0]], device=DEV), torch.full((1,), 0.9, device=DEV))
    w2c = np.zeros((cams, 3, 4), np.float32)
    w2c[:, 0, 0] = w2c[:, 1, 1] = w2c[:, 2, 2] = 1.0
    w2c[:, 2, 3] = 6.0
    intr = np.tile(np.array([w, w, w / 2, h / 2], np.float32), (cams, 1))
    return sc, icgs.Cameras(w, h, intr, w2c.reshape(-1, 12))


@pytest.mark.parametrize("K", [1, 3, 4, 7])
def test_empty_tiles(icgs, K):
    sc, cm = _one_gaussian(icgs, 2, 77, 51)
    targets = torch.rand((2, 51, 77, K), device=DEV)
    coeffs, status, chol = icgs.colorize(sc, cm, targets, 0)
    assert bool(torch.isfinite(coeffs).all()) and int(status[0]) != 1
    junk = torch.full((2, 51, 77, K), 7.0, device=DEV)  # what a fresh image may find in its memory
    del junk
    img = icgs.render(sc, cm, torch.ones((1, 1, K), device=DEV), 0)
    corner = torch.zeros((2, 51, 77, K), dtype=torch.bool, device=DEV)
    corner[:, :16, :16] = True  # the Gaussian is at the centre
    assert float(img.max()) > 0.0 and not bool(img[corner].any())
    junk = torch.full((2, 51, 77, K), 7.0, device=DEV)
    del junk
    gt, go = icgs.colorize_backward(sc, cm, targets, 0, coeffs, chol, torch.ones_like(coeffs))
    assert bool((gt != 0.0).any()) and not bool(gt[corner].any())
    targets[1, 3, 2, K - 1] = float("nan")
    for call in (lambda: icgs.colorize(sc, cm, targets, 0),
                 lambda: icgs.colorize_refine(sc, cm, targets, 0, coeffs.clone(), chol, 1)):
        with pytest.raises(icgs.IcgsError):
            call()


def _best_ms(f, ms):
    f()
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, ms(a, b))
    return best


def test_empty_tiles_cost_their_bytes(icgs):
    """The walks of 40 nearly empty views against the same bytes read or written once by torch: at most three times
    as long (a CTA per tile, its list's bounds, then its pixels)."""
    sc, cm = _one_gaussian(icgs, 40, W, H)
    targets = torch.rand((40, H, W, 3), device=DEV)
    coeffs = torch.ones((1, 1, 3), device=DEV)
    image = torch.empty_like(targets)
    elapsed = lambda a, b: a.elapsed_time(b)
    read, write = _best_ms(targets.sum, elapsed), _best_ms(image.zero_, elapsed)
    icgs.set_stage_timing(True)
    try:
        stage = lambda a, b: icgs.last_stage_ms()["blend"]
        accumulate = _best_ms(lambda: icgs.colorize(sc, cm, targets, 0), stage)
        render = _best_ms(lambda: icgs.render(sc, cm, coeffs, 0), stage)
    finally:
        icgs.set_stage_timing(False)
    print(f"read {read:.3f} accumulate {accumulate:.3f}; write {write:.3f} render {render:.3f} ms")
    assert accumulate <= 3.0 * read
    assert render <= 3.0 * write
