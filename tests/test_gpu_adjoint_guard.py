"""A Gaussian whose adjoint terms are not finite, or whose gain g = a . t + beta overflows FP32 although a, beta and
the targets are finite, spoils the gradients of the pixels that it contributes to and of the Gaussians with weight
there, and no others: the walks by 8-lane groups visit it at more pixels than those, with weight 0."""
import numpy as np
import pytest

from paper_2604_17155_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
Y0 = 0.28209479177387814


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("kind", ["overflow", "inf", "nan"])
def test_a_spoilt_gain_stays_with_its_pixels(K, kind):
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs

    sc = W.cluster_scene(3000, 461, radius=1.5, log_scale_mean=-3.6, log_scale_std=0.4)
    cams = W.hemisphere_cameras(3, 4.0, 77, 51, 50.0)
    gs, gc = icgs.Scene.from_workload(sc, DEV), icgs.Cameras.from_workload(cams)
    targets = torch.full((3, 51, 77, K), 8.0, device=DEV)
    coeffs, status, chol = icgs.colorize(gs, gc, targets, 0)
    weight = icgs.accumulate(gs, gc, torch.ones((3, 51, 77, 1), device=DEV), 0)[:, -1]
    seen = torch.nonzero((weight > 0.5) & (weight < 3.0)).flatten()
    picked = seen[torch.arange(3, device=DEV) * (len(seen) // 3)]
    # a = Y0 u, u = A^-1 dL/dc and A = w (Y0^2 + lambda): a = 8e37 where u = 2.8e38 is finite and a t = 6.4e38 is not
    amount = {"overflow": 8e37 / Y0, "inf": float("inf"), "nan": float("nan")}[kind]
    grad = torch.tensor(np.random.default_rng(462).standard_normal((sc.n, 1, K)), dtype=torch.float32, device=DEV)
    grad[picked] = 0.0
    coeffs[picked] = 0.0  # beta = 0
    spoilt = grad.clone()
    A = (weight[picked] * (Y0 * Y0 + 1e-5)).float()
    spoilt[picked] = (amount * A)[:, None, None] if kind == "overflow" else amount
    ref_t, ref_o = icgs.colorize_backward(gs, gc, targets, 0, coeffs, chol, grad)
    got_t, got_o = icgs.colorize_backward(gs, gc, targets, 0, coeffs, chol, spoilt)
    # the pixels that a picked Gaussian contributes to, and the Gaussians with weight in one of them
    alone = torch.zeros((sc.n, 1, 1), device=DEV)
    alone[picked] = 1.0
    touched = icgs.render(gs, gc, alone, 0) != 0.0
    near = icgs.accumulate(gs, gc, touched.float(), 0)[:, 1] != 0.0
    clean_px = ~touched[..., 0]
    assert 0 < int(clean_px.sum()) < clean_px.numel() and 0 < int(near.sum()) < sc.n // 2
    assert bool(torch.isfinite(ref_t).all()) and bool(torch.isfinite(ref_o).all())
    assert not bool(torch.isfinite(got_o[picked]).all())  # the case is what it is meant to be
    assert torch.equal(got_t[clean_px], ref_t[clean_px])
    # sums over tiles by atomics: FP32 sums of the same terms in another order
    scale = float(ref_o.abs().max())
    assert bool(torch.isfinite(got_o[~near]).all())
    assert float((got_o[~near] - ref_o[~near]).abs().max()) <= 1e-5 * scale
