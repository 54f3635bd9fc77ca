"""FP32 beamforming with the antennas split over a cluster of CTAs (three TF32 products per FP32 product) against the
FP64 oracle, at the edges of its tiles: 1, 2 and 4 CTAs per tile, a last CTA with few antennas, odd subcarrier and beam
counts (8-byte output rows), a last tile of one subcarrier, and buffers that are not 16-byte aligned.

Tolerance: an operand keeps all but 2^-23 of itself, the dropped lo x lo product is below 2^-22, and an accumulator
takes at most 8 truncated steps (2^-23 of the running sum each): 8 * 2^-23 + 3 * 2^-22 = 1.7e-6 of |A||B|; asserted
as 2e-6 of the norm, over all values and for every beam row of the largest shapes' worst row at 1e-5."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rx,n_beams,n_sc,offset", [
    (32, 33, 129, 0), (33, 40, 300, 0), (64, 63, 257, 0), (65, 64, 128, 0), (97, 34, 255, 0), (128, 64, 333, 1),
    (129, 48, 130, 0), (193, 64, 100, 0), (256, 64, 385, 1), (256, 33, 1, 0), (40, 17, 3276, 0)], ids=lambda v: str(v))
def test_split_antenna_beamforming(orc, n_rx, n_beams, n_sc, offset):
    n = 1
    rng = np.random.default_rng(n_rx * 1000 + n_beams + n_sc)
    cell = synth.SMALL_FP32.with_(n_rx=n_rx, n_beams=n_beams, n_layers=1, n_sc=n_sc, n_fft=4096)
    rx = host.Receiver(host.cfg_for(cell), max_slots=n)
    X = (rng.standard_normal((n, 14, n_rx, n_sc)) + 1j * rng.standard_normal((n, 14, n_rx, n_sc))).astype(np.complex64)
    W = ((rng.standard_normal((n_rx, n_beams)) + 1j * rng.standard_normal((n_rx, n_beams))) / np.sqrt(n_rx)).astype(np.complex64)
    flat = torch.zeros(X.size + offset, dtype=torch.complex64, device="cuda")
    flat[offset:] = torch.from_numpy(X.reshape(-1)).cuda()
    out = torch.full((n * 14 * n_sc * n_beams + offset,), float("nan"), dtype=torch.complex64, device="cuda")
    beam = out[offset:].view(n, 14, n_sc, n_beams)
    rx.beamform(flat[offset:].view(X.shape), host.beam_tensor(W), beam)
    torch.cuda.synchronize()
    Y = beam.cpu().numpy().astype(np.complex128)
    ref = orc.beamform(X[0].astype(np.complex128), W.astype(np.complex128))
    err = np.linalg.norm(Y[0] - ref) / np.linalg.norm(ref)
    row = np.abs(Y[0] - ref).max(axis=-1) / np.linalg.norm(ref, axis=-1)
    assert err < 2e-6, err
    assert row.max() < 1e-5, row.max()
    rx.close()
