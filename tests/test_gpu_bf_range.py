"""FP32 beamforming on split TF32 operands at the ends of the FP32 range, antennas split over 1, 2 and 4 CTAs: values next to
FLT_MAX, infinities and NaN in one sample or one weight, and all samples small.

Finite values: 2e-6 of the norm, as for ordinary ones (an operand keeps all but 2^-23 of itself, at most 8 truncated
steps); small samples from 2^-114 up, below which the lower part of a sample leaves the normal range. An infinite sample
gives, in its subcarrier and symbol only, the infinities and NaN of the FP32 sum."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu

SHAPES = [(64, 40, 257), (128, 33, 129), (256, 64, 130)]


def cell(n_rx, n_beams, n_sc):
    return host.Receiver(host.cfg_for(synth.SMALL_FP32.with_(n_rx=n_rx, n_beams=n_beams, n_layers=1, n_sc=n_sc, n_fft=4096)),
                         max_slots=1)


def inputs(n_rx, n_beams, n_sc, scale):
    g = torch.Generator(device="cuda")
    g.manual_seed(n_rx)
    X = torch.view_as_complex((torch.randn((1, 14, n_rx, n_sc, 2), generator=g, device="cuda") * scale))
    W = torch.view_as_complex(torch.randn((n_rx, n_beams, 2), generator=g, device="cuda") / (10.0 * n_rx ** 0.5))
    return X, W


def reference(X, W):
    return torch.einsum("nsrk,rb->nskb", X.to(torch.complex128), W.to(torch.complex128).conj())


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("value", [3.4028e38, float(np.finfo(np.float32).max), -float(np.finfo(np.float32).max)])
def test_a_sample_next_to_the_largest_float(shape, value):
    rx = cell(*shape)
    X, W = inputs(*shape, 1e30)
    X[0, 3, shape[0] - 1, 7] = value
    y, ref = rx.beamform(X, W), reference(X, W)
    assert bool(torch.isfinite(torch.view_as_real(y)).all())
    assert float((y - ref).norm() / ref.norm()) < 2e-6
    assert float((y[0, 3, 7] - ref[0, 3, 7]).norm() / ref[0, 3, 7].norm()) < 2e-6
    rx.close()


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan")])
def test_a_sample_that_is_not_finite(shape, value):
    rx = cell(*shape)
    X, W = inputs(*shape, 1.0)
    clean = rx.beamform(X, W).clone()
    X[0, 5, 2, 11] = complex(value, 0.5)
    y = rx.beamform(X, W)
    # the FP32 sum: value * Re W + ..., value * (-Im W) + ...
    w = W[2].conj()
    want = torch.view_as_complex(torch.stack([value * w.real, value * w.imag], -1))
    got = y[0, 5, 11]
    for a, b in ((got.real, want.real), (got.imag, want.imag)):
        assert bool(((a == b) | (a.isnan() & b.isnan())).all())
    y[0, 5, 11] = clean[0, 5, 11]
    assert torch.equal(y, clean)
    rx.close()


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_a_weight_that_is_infinite(shape):
    rx = cell(*shape)
    X, W = inputs(*shape, 1.0)
    clean = rx.beamform(X, W).clone()
    W[1, 4] = complex(float("inf"), 0.25)
    y = rx.beamform(X, W)
    assert torch.equal(y[..., 4].real, float("inf") * X[:, :, 1].real)
    assert torch.equal(y[..., 4].imag, float("inf") * X[:, :, 1].imag)
    y[..., 4] = clean[..., 4]
    assert torch.equal(y, clean)
    rx.close()


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("exponent", [-110, -60, 60, 120])
def test_small_and_large_samples(shape, exponent):
    rx = cell(*shape)
    X, W = inputs(*shape, 2.0 ** exponent)
    y, ref = rx.beamform(X, W), reference(X, W)
    assert float((y - ref).norm() / ref.norm()) < 2e-6
    rx.close()
