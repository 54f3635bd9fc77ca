"""The learned estimator's backward pass on given activations against the same sums in 64 bits, where every CTA takes
several tiles: the input gradients that it leaves in its work buffer, element by element.

The activations are random and half of them zero, so an element whose ReLU mask comes from another tile than its own is
wrong by its whole value.

Tolerance: an input gradient is a sum of at most 192 products, in at most 36 truncated tensor-core steps (2^-23 of the
running sum each) or 12 FMAs, of operands split to 2^-24 of themselves; with 48 * 2^-23 < 6e-6 of the sum of the products'
magnitudes for each of the layers so far. Truncation shrinks: half of a unit in the last place (2^-25 to 2^-24 of the
sum) is lost on average in each step that meets a sum of full size. With the parts of the split operand taken smallest
first these are 12 steps a layer, 12 * 2^-25 = 3.6e-7 of the norm where a step loses as little as it can (36 steps:
1.1e-6)."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import denoiser as D

pytestmark = pytest.mark.gpu

CH, DIL = (2, 32, 32, 32, 2), (1, 8, 16, 1)


def layers(p):
    """[(weights, first weight, first bias)] of the packed parameters."""
    out, o = [], 0
    for k in range(4):
        n = CH[k] * CH[k + 1] * 9
        out.append((p[o:o + n].reshape(CH[k + 1], CH[k], 3, 3), o, o + n))
        o += n + CH[k + 1]
    return out


def shifted(a, d):
    """a[.., x + d], zero outside the grid."""
    z = torch.zeros_like(a)
    w = a.shape[-1]
    if abs(d) < w:
        if d >= 0:
            z[..., :w - d] = a[..., d:]
        else:
            z[..., -d:] = a[..., :d]
    return z


def input_grad(g, W, dil):
    """[n, co, 2, w] -> [n, ci, 2, w]"""
    out = torch.zeros((g.shape[0], W.shape[1], 2, g.shape[-1]), dtype=g.dtype, device=g.device)
    for kw in range(3):
        s = shifted(g, -(kw - 1) * dil)
        for h in range(2):
            for r in range(2):
                out[:, :, r] += torch.einsum("nox,oi->nix", s[:, :, h], W[:, :, r - h + 1, kw])
    return out


def weight_grad(g, a, dil):
    """sum over grids and subcarriers -> [co, ci, 3, 3]"""
    out = torch.zeros((g.shape[1], a.shape[1], 3, 3), dtype=g.dtype, device=g.device)
    for kw in range(3):
        s = shifted(a, (kw - 1) * dil)
        for h in range(2):
            for r in range(2):
                out[:, :, r - h + 1, kw] += torch.einsum("nox,nix->oi", g[:, :, h], s[:, :, r])
    return out


def inputs(n, w, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    p = torch.from_numpy(D.init_params(seed)).cuda().to(torch.bfloat16)
    return dict(n=n, w=w, p=p, x=rnd(n, 2, 2, w).to(torch.bfloat16), y=rnd(n, 2, 2, w), target=rnd(n, 2, 2, w),
                acts=rnd(3, n, 32, 2, w).relu().to(torch.bfloat16))


def backward(c):
    n, w = c["n"], c["w"]
    grad = torch.full((D.PARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    work = torch.full((2, n, w, 64), float("nan"), device="cuda")
    B.pusch_cnn_backward(n, w, c["x"], c["acts"], c["p"], c["y"], c["target"], grad, loss, work,
                         torch.zeros(D.PARAMS, dtype=torch.bfloat16, device="cuda"))
    torch.cuda.synchronize()
    return grad, loss, work


@pytest.mark.parametrize("n,w", [(930, 100), (311, 300), (1300, 128)])
def test_input_gradients_with_several_tiles_per_cta(n, w):
    c = inputs(n, w, n + w)
    _, _, work = backward(c)
    P = layers(c["p"].double())
    g = 2.0 * (c["y"].double() - c["target"].double()) / (4.0 * n * w)
    mag = g.abs()
    # layer 4's input gradient is overwritten by layer 2's; layer 3's lies in the first half
    for k, where in ((3, None), (2, work[0]), (1, work[1])):
        on = c["acts"][k - 1].double() > 0
        g = input_grad(g, P[k][0], DIL[k]) * on
        mag = input_grad(mag, P[k][0].abs(), DIL[k]) * on
        if where is not None:
            got = where.reshape(n, w, 2, 32).permute(0, 3, 2, 1).double()
            off = (got - g).abs()
            assert bool((off <= 6e-6 * (4 - k) * mag).all()), (k, float((off / mag.clamp(min=1e-300)).max()))


def test_input_gradients_shrink_by_the_steps_of_the_largest_part():
    n, w = 64, 96
    c = inputs(n, w, 5)
    _, _, work = backward(c)
    P = layers(c["p"].double())
    g = 2.0 * (c["y"].double() - c["target"].double()) / (4.0 * n * w)
    for k, where in ((3, None), (2, work[0]), (1, work[1])):
        g = input_grad(g, P[k][0], DIL[k]) * (c["acts"][k - 1] > 0)
        if where is not None:
            got = where.reshape(n, w, 2, 32).permute(0, 3, 2, 1).double()
            assert float((got - g).norm() / g.norm()) < 3.6e-7 * (3 - k), k


@pytest.mark.parametrize("n,w", [(4096, 64), (1500, 300)])
def test_weight_gradients_do_not_shrink_with_the_number_of_tiles(n, w):
    """Layers 3 and 2: the projection on the 64-bit gradient, from which random rounding is absent. A tile's sum meets
    8 steps of the largest part, layer 2's gradient also carries the shrinking of its input gradient (above)."""
    c = inputs(n, w, 7)
    grad, _, _ = backward(c)
    P = layers(c["p"].double())
    g = 2.0 * (c["y"].double() - c["target"].double()) / (4.0 * n * w)
    for k, steps in ((3, None), (2, 8), (1, 12 + 8)):
        a = c["acts"][k - 1].double()
        if steps is not None:
            ref = weight_grad(g, a, DIL[k]).reshape(-1)
            got = grad[P[k][1]:P[k][2]].double()
            shrink = float((got - ref) @ ref / (ref @ ref))
            assert abs(shrink) < steps * 2.0 ** -25, (k, shrink)
        g = input_grad(g, P[k][0], DIL[k]) * (a > 0)
