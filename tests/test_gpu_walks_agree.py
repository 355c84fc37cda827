"""The walks by 8-lane groups take the decisions and weights of the one-pixel walks bit for bit: images of up to four
channels against the same channels of an eight-channel render, and the number of contributing (pixel, Gaussian) pairs
over every accumulation walk. On scenes where the groups' list test is tightest: needles, opacities just above 1/255,
Gaussians larger than the image and smaller than a pixel, and opaque stacks, with ragged edges and lists of several
batches."""
import numpy as np
import pytest

from paper_2604_17155_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
N, CAMS, WIDTH, HEIGHT = 12_000, 4, 141, 93


@pytest.fixture(scope="module")
def icgs():
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs as I
    I.load()
    return I


def _scene(icgs, kind):
    rng = np.random.default_rng(sum(map(ord, kind)))
    means = rng.normal(0.0, 0.7, (N, 3))
    scales = np.exp(rng.normal(-3.6, 0.5, (N, 3)))
    opacity = 1.0 / (1.0 + np.exp(-rng.normal(0.5, 2.0, N)))
    if kind == "needles":  # a hundred to a hundred thousand times as long as thick, in every direction
        scales = np.exp(rng.uniform(-11.0, -6.0, (N, 3)))
        scales[np.arange(N), rng.integers(0, 3, N)] = np.exp(rng.uniform(-1.5, 1.0, N))
    elif kind == "faint":  # a support of a fraction of a pixel to a few, where the threshold decides
        opacity = (1.0 / 255.0) * (1.0 + np.exp(rng.uniform(np.log(1e-6), np.log(3.0), N)))
    elif kind == "faint_needles":
        scales = np.exp(rng.uniform(-11.0, -6.0, (N, 3)))
        scales[np.arange(N), rng.integers(0, 3, N)] = np.exp(rng.uniform(-1.5, 1.0, N))
        opacity = (1.0 / 255.0) * (1.0 + np.exp(rng.uniform(np.log(1e-6), np.log(3.0), N)))
    elif kind == "large":
        scales = np.exp(rng.normal(0.5, 1.0, (N, 3)))
        opacity = rng.uniform(0.004, 0.03, N)
    elif kind == "specks":
        scales = np.exp(rng.uniform(-12.0, -7.0, (N, 3)))
    elif kind == "opaque":
        opacity = rng.uniform(0.9, 1.0, N)
    f = lambda x: torch.tensor(x, dtype=torch.float32, device=DEV)
    return icgs.Scene(f(means), f(scales), f(rng.normal(size=(N, 4))), f(opacity))


KINDS = ["plain", "needles", "faint", "faint_needles", "large", "specks", "opaque"]


@pytest.mark.parametrize("kind", KINDS)
def test_images(icgs, kind):
    gs = _scene(icgs, kind)
    gc = icgs.Cameras.from_workload(W.hemisphere_cameras(CAMS, 4.0, WIDTH, HEIGHT, 50.0))
    coeffs = torch.tensor(W.sh_coefficients(N, 1, 8, seed=491), dtype=torch.float32, device=DEV)
    ref = icgs.render(gs, gc, coeffs, 1)
    assert bool((ref != 0.0).any())
    for K in (1, 2, 3, 4):
        img = icgs.render(gs, gc, coeffs[..., :K].contiguous(), 1)
        assert torch.equal(img, ref[..., :K]), K


@pytest.mark.parametrize("kind", KINDS)
def test_contributing_pairs(icgs, kind):
    gs = _scene(icgs, kind)
    gc = icgs.Cameras.from_workload(W.hemisphere_cameras(CAMS, 4.0, WIDTH, HEIGHT, 50.0))
    targets = torch.rand((CAMS, HEIGHT, WIDTH, 16), device=DEV, generator=torch.Generator(DEV).manual_seed(492))

    def pairs(t):
        icgs.colorize(gs, gc, t.contiguous(), 0)
        return icgs.last_stats()["contrib_pairs"]

    ref = pairs(targets[..., :8])  # one pixel a thread
    assert ref > 0
    for K in (1, 2, 3, 7):  # 4x8 and 8x4 blocks
        assert pairs(targets[..., :K]) == ref, K
    assert pairs(targets.half()) == ref  # 4x4 blocks, tensor cores
