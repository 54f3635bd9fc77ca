"""The learned estimator's kernels at the edges of their tiles (256 subcarriers, 206 outputs where a grid takes several)
against the FP64 oracle with bfloat16 rounding at the same points: widths of one subcarrier, just below, at and above a
tile, one output in the last tile, odd widths, and more grids than tiles in flight. Bars: those of the other CNN tests
(one bfloat16 rounding, 2^-9, per activation; the last layer's sums in FP32), and no subcarrier's output off by more
than ten such roundings of the RMS, so that a seam between tiles shows."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import denoiser as D

pytestmark = pytest.mark.gpu


def nrel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(b.ravel()), 1e-300))


@pytest.mark.parametrize("n,w", [(1, 1), (2, 25), (1, 255), (3, 256), (1, 257), (1, 412), (2, 413), (1, 619), (700, 33)])
def test_tile_edges(orc, n, w):
    rng = np.random.default_rng(n * 1000 + w)
    p = D.init_params(seed=n)
    p[-(2 * 32 * 9 + 2):] *= 10.0
    x = rng.standard_normal((n, 2, 2, w)).astype(np.float32)
    tgt = rng.standard_normal((n, 2, 2, w)).astype(np.float32)
    pb = torch.from_numpy(p).cuda().to(torch.bfloat16)
    xb = torch.from_numpy(x).cuda().to(torch.bfloat16)
    y = torch.full((n, 2, 2, w), float("nan"), device="cuda")
    acts = torch.full((3, n, 32, 2, w), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.pusch_cnn_forward(n, w, xb, pb, y, acts)
    grad = torch.full((D.PARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    work = torch.full((2 * n * 32 * 2 * w,), float("nan"), device="cuda")
    wflip = torch.zeros(D.PARAMS, dtype=torch.bfloat16, device="cuda")
    B.pusch_cnn_backward(n, w, xb, acts, pb, y, torch.from_numpy(tgt).cuda(), grad, loss, work, wflip)
    torch.cuda.synchronize()
    yo, ao = orc.cnn_forward(p, x, bf16=True)
    yg = y.cpu().numpy()
    assert nrel(yg, yo) < 2e-3
    assert np.abs(yg - yo).max() < 10 * 2.0 ** -9 * np.sqrt(np.mean(np.square(yo)))
    assert nrel(acts.float().cpu().numpy(), ao) < 2e-3
    lo, go = orc.cnn_loss_grad(p, x, tgt, bf16=True)
    assert abs(float(loss) - lo) < 2e-3 * lo
    assert nrel(grad.cpu().numpy(), go) < 5e-3
