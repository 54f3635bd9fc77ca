"""The tensor-core FFT's stores: every remainder of the FFT shift modulo eight, the widths at the ends of the
range, and an output whose base allows no 16-byte stores, through pusch_ofdm_fft (Section II, "OFDM dem.").

Against the DFT in 64 bits at the FP16 bar of the mixed form: FP16 intermediate and output, two roundings of
at most 2^-11 each and the DFT matrix's own, under 3 x 2^-11 = 1.5e-3 per row norm."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu


def _rx(n_sc):
    cell = synth.CellConfig("fft", n_rx=8, n_fft=4096, n_sc=n_sc, n_beams=8, n_layers=2, qam_bits=2, snr_db=30.0,
                            channel="pdp", beam="dft", in_fp16=True, seed=3)
    return host.Receiver(host.cfg_for(cell, B.PUSCH_FORM_MIXED), max_slots=1)


def _time(n_sc):
    rng = np.random.default_rng(n_sc)
    return (rng.standard_normal((1, 14, 8, 4096, 2)) * 0.02).astype(np.float16)


@pytest.mark.parametrize("n_sc", [1200, 1202, 1204, 1206, 1208, 1210, 1212, 1214, 12, 4092, 4095])
def test_fft_shift_remainders(n_sc):
    t16 = _time(n_sc)
    rx = _rx(n_sc)
    f = rx.ofdm_fft(torch.from_numpy(t16).cuda()).cpu().numpy().astype(np.float64)
    assert np.all(f[..., n_sc:] == 0)
    x = t16[..., 0].astype(np.float64) + 1j * t16[..., 1].astype(np.float64)
    ref = np.fft.fft(x, axis=-1)[..., (np.arange(n_sc) - n_sc // 2) % 4096]
    got = f[..., 0, :n_sc] + 1j * f[..., 1, :n_sc]
    rel = np.linalg.norm(got - ref, axis=-1) / np.linalg.norm(ref, axis=-1)
    assert np.max(rel) < 1.5e-3
    rx.close()


def test_fft_output_on_a_two_byte_boundary():
    rx = _rx(3276)
    t = torch.from_numpy(_time(3276)).cuda()
    want = rx.ofdm_fft(t)
    raw = torch.full((want.numel() + 1,), 7.0, dtype=torch.float16, device="cuda")
    out = raw[1:].view(want.shape)
    rx.ofdm_fft(t, freq=out)
    torch.cuda.synchronize()
    assert torch.equal(out, want) and float(raw[0]) == 7.0
    rx.close()
