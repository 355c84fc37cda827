"""The order in which Gaussians enter the binning, by cells of space or as given, and the scan of the tile counts, in one
CTA or in three kernels: which call takes which, and that the images are the same bits."""
import pytest

from paper_2604_17155_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def icgs():
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs as I
    I.load()
    return I


def _scene(icgs, n, seed, n_cams, w, h):
    sc = W.cluster_scene(n, seed, radius=1.5, log_scale_mean=-3.6, log_scale_std=0.4)
    return icgs.Scene.from_workload(sc, DEV), icgs.Cameras.from_workload(W.hemisphere_cameras(n_cams, 4.0, w, h, 50.0))


def test_both_orders_and_both_scans_give_the_same_images(icgs):
    """128 views of 160 x 112: ordered, 8,960 counts (three kernels, the last block of 1,024 partly filled); 10 at a time:
    input order, 700 counts (one CTA, one round partly filled), and 116: ordered, 8,120 (one CTA, eight rounds)."""
    n, w, h = 100_003, 160, 112
    gs, gc = _scene(icgs, n, 481, 128, w, h)
    coeffs = torch.tensor(W.sh_coefficients(n, 1, 3, seed=482), dtype=torch.float32, device=DEV)
    tiles = (w // 16) * (h // 16)
    assert 128 * tiles > 8192 > 116 * tiles
    whole = icgs.render(gs, gc, coeffs, 1)
    three = icgs.last_stats()["launches"]
    assert torch.equal(icgs.render(gs, gc.subset(list(range(116))), coeffs, 1), whole[:116])
    assert icgs.last_stats()["launches"] == three - 2  # the scan
    for j in range(0, 120, 10):
        assert torch.equal(icgs.render(gs, gc.subset(list(range(j, j + 10))), coeffs, 1), whole[j:j + 10])
        assert icgs.last_stats()["launches"] == three - 8  # and the order


@pytest.mark.parametrize("n,many,few,w,h", [(30_000, 100, 2, 1600, 1060), (400_000, 16, 3, 3840, 2160)])
def test_many_tiles_are_binned_in_cell_order(icgs, n, many, few, w, h):
    gs, gc = _scene(icgs, n, 483, many, w, h)
    coeffs = torch.ones((n, 1, 1), device=DEV)
    icgs.render(gs, gc, coeffs, 0)
    ordered = icgs.last_stats()["launches"]
    icgs.render(gs, gc.subset(list(range(few))), coeffs, 0)
    assert icgs.last_stats()["launches"] == ordered - 6


def test_few_views_are_binned_in_input_order(icgs):
    """Two million Gaussians in eight small views take the launches of one view."""
    n = 2_000_000
    gs, gc = _scene(icgs, n, 484, 8, 64, 64)
    coeffs = torch.ones((n, 1, 1), device=DEV)
    icgs.render(gs, gc, coeffs, 0)
    eight = icgs.last_stats()["launches"]
    icgs.render(gs, gc.subset([0]), coeffs, 0)
    assert icgs.last_stats()["launches"] == eight
