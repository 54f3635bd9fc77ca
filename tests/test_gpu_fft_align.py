"""The tensor-core FFT into buffers at every distance from a 16-byte boundary: the values of the aligned call, nothing
written beside the planes, and about its time (the stores stay 16 bytes wide; value by value they took three times as
long). Widths around the ends of the range, so that octets cross the planes' ends and the transform's."""
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu


def receiver(n_sc, n_rx=8):
    cell = synth.CellConfig("fft", n_rx=n_rx, n_fft=4096, n_sc=n_sc, n_beams=8, n_layers=2, qam_bits=2, snr_db=30.0,
                            channel="pdp", beam="dft", in_fp16=True, seed=3)
    return host.Receiver(host.cfg_for(cell, B.PUSCH_FORM_MIXED), max_slots=1)


def samples(n_rx, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn((1, 14, n_rx, 4096, 2), generator=g, device="cuda") * 0.02).half()


@pytest.mark.parametrize("n_sc", [2, 12, 13, 127, 1200, 1203, 1206, 3275, 3276, 4033, 4092, 4095, 4096])
def test_fft_at_every_alignment(n_sc):
    rx = receiver(n_sc)
    t = samples(8, n_sc)
    want = rx.ofdm_fft(t)
    raw = torch.empty(want.numel() + 24, dtype=torch.float16, device="cuda")
    for off in range(8):
        raw.fill_(7.0)
        a = 8 + off
        rx.ofdm_fft(t, freq=raw[a:a + want.numel()].view(want.shape))
        assert torch.equal(raw[a:a + want.numel()].view(want.shape), want), off
        assert bool((raw[:a] == 7.0).all()) and bool((raw[a + want.numel():] == 7.0).all()), off
    rx.close()


def test_an_unaligned_output_costs_little():
    rx = receiver(3276, 64)
    t = samples(64, 1)
    want = rx.ofdm_fft(t)
    raw = torch.zeros(want.numel() + 8, dtype=torch.float16, device="cuda")

    def us(off):
        out = raw[off:off + want.numel()].view(want.shape)
        times = []
        for _ in range(20):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                rx.ofdm_fft(t, freq=out)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times)[10]

    us(0)
    aligned = us(0)
    assert us(4) < 1.7 * aligned and us(1) < 1.7 * aligned
    rx.close()
