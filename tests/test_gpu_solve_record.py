"""The solve record: its A against the packed sums and its factor against A, for Gaussians solved in FP32, re-folded and
in FP64, where the shared memory of a solve holds the bases of a re-fold, the factor and the record in turn; with one
and with several groups of channels."""
import numpy as np
import pytest

from paper_2604_17155_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("L", [1, 2, 3])
@pytest.mark.parametrize("K", [3, 9])
@pytest.mark.parametrize("way", ["plain", "mixed", "refold", "fp64", "refold_fp64"])
def test_record(L, K, way):
    from paper_2604_17155_gb300 import build as B
    B.build()
    from paper_2604_17155_gb300 import icgs

    n, cams = 3001, 40
    sc = W.cluster_scene(n, 501, radius=1.5, log_scale_mean=-3.6, log_scale_std=0.4)
    gs = icgs.Scene.from_workload(sc, DEV)
    gc = icgs.Cameras.from_workload(W.hemisphere_cameras(cams, 4.0, 96, 72, 50.0))
    targets = torch.rand((cams, 72, 96, K), device=DEV, generator=torch.Generator(DEV).manual_seed(502))
    precision = "plain" if way == "plain" else "mixed"
    # pivot ratios lie below 1: thresholds above send every Gaussian there
    kw = dict(refold_tau=2.0 if "refold" in way else 0.0,
              cond_tau=2.0 if way == "fp64" else (200.0 if way == "refold_fp64" else 1e-7))
    coeffs, status, record = icgs.colorize(gs, gc, targets, L, precision=precision, **kw)
    stats = icgs.last_stats()
    sums = icgs.accumulate(gs, gc, targets, L, precision=precision).cpu().numpy()
    b = (L + 1) ** 2
    P = b * (b + 1) // 2
    w = sums[:, -1]
    seen = w > 0
    st = status.cpu().numpy()
    assert (st[seen] == (2 if "fp64" in way else 0)).mean() > 0.98 and (stats["refold"] > 0) == ("refold" in way)
    rows, cols = np.triu_indices(b)
    A = np.zeros((n, b, b))
    A[:, rows, cols] = sums[:, :P]
    A[:, cols, rows] = sums[:, :P]
    lam = np.concatenate([[x] * (2 * l + 1) for l, x in enumerate([1e-5, 1e-4, 1e-3, 1e-2][: L + 1])])
    A[:, range(b), range(b)] += w[:, None] * lam
    rec = record.cpu().numpy().astype(np.float64)
    low = np.tril_indices(b)
    got, fac = np.zeros((n, b, b)), np.zeros((n, b, b))
    got[:, low[0], low[1]] = rec[:, P:2 * P] + rec[:, 2 * P:]
    fac[:, low[0], low[1]] = rec[:, :P]
    scale = w[:, None, None] + 1e-30
    # the sums of V differ between two calls by the order of their atomics (2^-22 of w); PLAIN folds in FP32
    assert np.abs((got - np.tril(A))[seen] / scale[seen]).max() <= (2e-5 if way == "plain" else 2e-6)
    whole = np.abs(np.tril(fac @ fac.transpose(0, 2, 1) - A) / scale)[seen]
    assert whole.max() <= 5e-5  # an FP32 Cholesky, backward stable
    assert not rec[~seen].any()
    assert bool(torch.isfinite(coeffs).all())
