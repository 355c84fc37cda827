"""The walks by 8-lane groups and the fold by block diagonals at the channel counts where their kernels and
layouts change, on ragged images whose tile lists take several batches, against the FP64 oracle; the colour
guard of the render; and the two orders in which Gaussians enter the binning. Tolerances are those of the
other parity files, set from the arithmetic: FP32 sums of some 10^3 terms (1e-4 after the solve), 11-bit
weights for 16-bit targets (2e-3)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2604_17155_gb300 import workloads as W

from _parity import (ADJ_TOL_O, ADJ_TOL_T, TOL_BF16, TOL_FP32, adjoint_flags, adjoint_report, coefficient_report,
                     to_np)

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


def _scene(n, seed, n_cams, w, h):
    sc = W.cluster_scene(n, seed, radius=1.5, log_scale_mean=-3.6, log_scale_std=0.4)
    return sc, W.hemisphere_cameras(n_cams, 4.0, w, h, 50.0)


def _gpu(icgs, sc, cams):
    return icgs.Scene.from_workload(sc, DEV), icgs.Cameras.from_workload(cams)


# FP32: every width of the group walk's sums (2, 4 and 8 values), then the first of the other walk and a
# second chunk of 1 and of 7 channels. 16 bits: the tensor-core operand's widths 16, 24, 32, 48 and 64, whole and
# padded.
@pytest.mark.parametrize("K,dtype", [(1, "f32"), (2, "f32"), (3, "f32"), (4, "f32"), (7, "f32"), (8, "f32"),
                                     (17, "f32"), (23, "f32"), (16, "bf16"), (17, "f16"), (21, "f16"), (24, "bf16"), (25, "f16"),
                                     (32, "bf16"), (33, "f16"), (48, "bf16"), (49, "f16"), (63, "bf16"), (64, "f16")])
def test_accumulate_widths(icgs, K, dtype):
    sc, cams = _scene(6000, 401, 6, 77, 51)
    rng = np.random.default_rng(402 + K)
    tt = torch.tensor(rng.uniform(0, 1, (cams.n, 51, 77, K)), device=DEV).to(
        {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dtype])
    lam = [1e-5]
    col = O.colorize(sc, cams, tt.double().cpu().numpy(), 0, lam)
    gs, gc = _gpu(icgs, sc, cams)
    c, status, chol = icgs.colorize(gs, gc, tt, 0, lam=lam)
    tol = TOL_FP32 if dtype == "f32" else TOL_BF16
    rep, err, checked = coefficient_report(to_np(c), col, tol=tol)
    print(K, dtype, rep, icgs.last_stats())
    assert rep["checked"] > 0
    assert rep["max_checked"] <= tol
    assert rep["bound_excess"] <= 0


# Block counts 2, 5 and 8 of the fold, with 1, 2 and 3 channels in its last group of three or four.
@pytest.mark.parametrize("L", [1, 2, 3])
@pytest.mark.parametrize("K", [1, 4, 5, 6, 9])
def test_fold_and_solve_channels(icgs, L, K):
    sc, cams = _scene(1501, 411 + L, 24, 96, 72)
    t = O.render(sc, cams, W.sh_coefficients(sc.n, L, K, seed=421 + L), L).astype(np.float32)
    col = O.colorize(sc, cams, t.astype(np.float64), L)
    gs, gc = _gpu(icgs, sc, cams)
    tt = torch.tensor(t, device=DEV)
    c, status, chol = icgs.colorize(gs, gc, tt, L)
    rep, err, checked = coefficient_report(to_np(c), col)
    print(L, K, rep)
    assert rep["checked"] > 0
    assert rep["max_checked"] <= TOL_FP32
    assert rep["bound_excess"] <= 0
    # the packed sums pass through the kept layout of G and back
    c2, s2, _ = icgs.solve(icgs.accumulate(gs, gc, tt, L), L)
    rep2, _, _ = coefficient_report(to_np(c2), col)
    assert rep2["max_checked"] <= TOL_FP32
    assert rep2["bound_excess"] <= 0


@pytest.mark.parametrize("K", [1, 2, 4])
def test_adjoint_channels(icgs, K):
    sc, cams = _scene(1500, 431, 8, 71, 45)
    L = 1
    t = O.render(sc, cams, W.sh_coefficients(sc.n, L, K, seed=432), L).astype(np.float32)
    t64 = t.astype(np.float64)
    col = O.colorize(sc, cams, t64, L)
    r = np.random.default_rng(433).standard_normal(col["c"].shape)
    gt_ref, go_ref = O.adjoint(sc, cams, t64, L, None, 2 * r * col["c"], col=col)
    flags = adjoint_flags(sc, cams, t64, col)
    gs, gc = _gpu(icgs, sc, cams)
    tt = torch.tensor(t, device=DEV)
    c, status, chol = icgs.colorize(gs, gc, tt, L)
    gcoef = torch.tensor(2 * r * col["c"], dtype=torch.float32, device=DEV)
    gt, go = icgs.colorize_backward(gs, gc, tt, L, torch.tensor(col["c"], dtype=torch.float32, device=DEV), chol, gcoef)
    rep = adjoint_report(to_np(gt), to_np(go), gt_ref, go_ref, col, flags)
    print(K, rep)
    assert rep["dt_max_clean"] <= ADJ_TOL_T
    assert rep["do_max_clean"] <= ADJ_TOL_O


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_nonfinite_colour_stays_with_its_pixels(icgs, K, value):
    """A Gaussian of non-finite colour spoils the pixels that it contributes to, and no other pixel."""
    sc, cams = _scene(3000, 441, 3, 77, 51)
    gs, gc = _gpu(icgs, sc, cams)
    clean = torch.tensor(W.sh_coefficients(sc.n, 0, K, seed=442), dtype=torch.float32, device=DEV)
    picked = [5, 900, 2222]
    alone = torch.zeros_like(clean)
    alone[picked] = 1.0
    spoilt = clean.clone()
    spoilt[picked] = value
    touched = icgs.render(gs, gc, alone, 0) != 0.0
    img, ref = icgs.render(gs, gc, spoilt, 0), icgs.render(gs, gc, clean, 0)
    assert 0 < int(touched.sum()) < touched.numel()
    assert not bool(torch.isfinite(img[touched]).any())
    assert torch.equal(img[~touched], ref[~touched])


def test_input_and_cell_order_give_the_same_images(icgs):
    """A call of more than 2^23 (camera, Gaussian) pairs visits the Gaussians by cells of space, a smaller one in
    input order (and scans its tile counts in one CTA): the images of both are the same bits."""
    n, cams_n = 100_003, 90
    sc, cams = _scene(n, 451, cams_n, 45, 33)
    gs, gc = _gpu(icgs, sc, cams)
    coeffs = torch.tensor(W.sh_coefficients(sc.n, 1, 3, seed=452), dtype=torch.float32, device=DEV)
    assert n * cams_n > 1 << 23 > n * 10
    whole = icgs.render(gs, gc, coeffs, 1)
    for j in range(0, cams_n, 10):
        part = icgs.render(gs, gc.subset(list(range(j, j + 10))), coeffs, 1)
        assert torch.equal(part, whole[j:j + 10])
