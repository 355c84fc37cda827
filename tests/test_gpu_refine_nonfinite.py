"""A refinement from coefficients that render to infinity: the residuals of those pixels spoil the Gaussians with
weight in the pixels' 8x4 blocks (the walk's unit of a sum), and no others."""
import pytest

from paper_2604_17155_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("K", [4, 7, 8])
def test_an_infinite_colour_stays_with_its_blocks(K):
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs

    w, h = 80, 64  # whole blocks
    sc = W.cluster_scene(3000, 471, radius=1.5, log_scale_mean=-3.6, log_scale_std=0.4)
    cams = W.hemisphere_cameras(3, 4.0, w, h, 50.0)
    gs, gc = icgs.Scene.from_workload(sc, DEV), icgs.Cameras.from_workload(cams)
    targets = torch.rand((3, h, w, K), device=DEV, generator=torch.Generator(DEV).manual_seed(472))
    coeffs, status, chol = icgs.colorize(gs, gc, targets, 0)
    picked = torch.tensor([5, 900, 2222], device=DEV)
    ref = icgs.colorize_refine(gs, gc, targets, 0, coeffs.clone(), chol, 1)
    spoilt = coeffs.clone()
    spoilt[picked] = float("inf")
    got = icgs.colorize_refine(gs, gc, targets, 0, spoilt, chol, 1)
    alone = torch.zeros((sc.n, 1, 1), device=DEV)
    alone[picked] = 1.0
    touched = (icgs.render(gs, gc, alone, 0) != 0.0).float().reshape(3, h // 4, 4, w // 8, 8)
    blocks = touched.amax((2, 4), keepdim=True).expand(3, h // 4, 4, w // 8, 8).reshape(3, h, w, 1).contiguous()
    near = icgs.accumulate(gs, gc, blocks, 0)[:, 1] != 0.0
    assert 0 < int(blocks.sum()) < blocks.numel() and 0 < int(near.sum()) < sc.n
    assert not bool(torch.isfinite(got[near]).all())  # the case is what it is meant to be
    assert bool(torch.isfinite(got[~near]).all())
    assert torch.allclose(got[~near], ref[~near], rtol=1e-4, atol=1e-4 * float(ref.abs().max()))
