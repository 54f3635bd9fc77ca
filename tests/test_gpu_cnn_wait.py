"""The learned estimator's kernels when a wait on their products expires. Every wait is on a barrier that nothing completes,
with a limit of 200 us; no address in the kernels depends on what a wait was for, and the products in flight are drained
before a CTA ends. The call returns in the time of the first wait (several tiles per CTA: the later ones are not waited
out), and calls after it give what calls before it gave."""
import time

import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import denoiser as D

pytestmark = pytest.mark.gpu


def buffers(n, w):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + w)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    return dict(x=rnd(n, 2, 2, w).to(torch.bfloat16), p=torch.from_numpy(D.init_params(3)).cuda().to(torch.bfloat16),
                y=torch.zeros((n, 2, 2, w), device="cuda"), target=rnd(n, 2, 2, w),
                acts=torch.zeros((3, n, 32, 2, w), dtype=torch.bfloat16, device="cuda"),
                grad=torch.zeros(D.PARAMS, device="cuda"), loss=torch.zeros(1, device="cuda"),
                work=torch.zeros(2 * n * 64 * w, device="cuda"))


def step(b, n, w):
    wflip = torch.zeros(D.PARAMS, dtype=torch.bfloat16, device="cuda")
    B.pusch_cnn_forward(n, w, b["x"], b["p"], b["y"], b["acts"])
    B.pusch_cnn_backward(n, w, b["x"], b["acts"], b["p"], b["y"], b["target"], b["grad"], b["loss"], b["work"], wflip)
    torch.cuda.synchronize()
    return [b[k].clone() for k in ("y", "acts", "loss", "grad")]


def selftest(b, n, w):
    B.pusch_selftest_cnn_wait(n, w, b["x"], b["p"], b["y"], b["acts"], b["target"], b["grad"], b["loss"], b["work"], 200)


@pytest.mark.parametrize("n,w", [(1, 40), (2000, 130)])
def test_expired_waits_end_the_call_and_leave_nothing_behind(n, w):
    b = buffers(n, w)
    before = step(b, n, w)
    t0 = time.time()
    selftest(b, n, w)
    torch.cuda.synchronize()
    assert time.time() - t0 < 5.0
    after = step(b, n, w)
    assert torch.equal(after[0], before[0]) and torch.equal(after[1], before[1])
    for u, v in zip(after[2:], before[2:]):                # sums over CTAs: FP32 additions in any order
        assert float((u - v).norm()) <= 1e-5 * float(v.norm())


def test_selftest_arguments():
    b = buffers(1, 8)
    for limit in (0, 1000001):
        with pytest.raises(B.PuschError) as ei:
            B.pusch_selftest_cnn_wait(1, 8, b["x"], b["p"], b["y"], b["acts"], b["target"], b["grad"], b["loss"],
                                      b["work"], limit)
        assert ei.value.code == B.PUSCH_ERR_ARG


@pytest.mark.parametrize("n,w", [(1, 40), (2000, 130)])
def test_expired_waits_show_in_the_outputs(n, w):
    """The backward pass runs on valid forward results, so what is not finite in its outputs it made so itself."""
    b = buffers(n, w)
    step(b, n, w)
    selftest(b, n, w)
    torch.cuda.synchronize()
    last = 2 * 32 * 9 + 2                                  # layer 4's gradients come from a kernel without waits
    assert bool(b["loss"].isnan().all()) and bool(b["grad"][:-last].isnan().all())
    assert not bool(b["grad"][-last:].isnan().any())
    assert bool(b["y"].isnan().all())
