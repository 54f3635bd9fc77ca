"""FP32 beamforming gives a slot the same values whatever batch it is in: the kernel is chosen by the cell alone. Cells with 17
to 32 beams on either side of every line of that choice, five slots in one call against the slots one by one and in
pairs, and the whole chain in one pass against its chunk runs."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rx,n_beams,n_sc", [
    (32, 24, 1023), (32, 24, 1025), (33, 17, 511), (33, 17, 513), (64, 31, 512), (64, 31, 601), (65, 20, 300),
    (128, 32, 601), (256, 32, 1200), (48, 33, 601), (48, 16, 1201)], ids=lambda v: str(v))
def test_slots_do_not_depend_on_their_batch(n_rx, n_beams, n_sc):
    n = 5
    rx = host.Receiver(host.cfg_for(synth.SMALL_FP32.with_(n_rx=n_rx, n_beams=n_beams, n_layers=1, n_sc=n_sc, n_fft=4096)),
                       max_slots=n)
    g = torch.Generator(device="cuda")
    g.manual_seed(n_rx + n_sc)
    X = torch.view_as_complex(torch.randn((n, 14, n_rx, n_sc, 2), generator=g, device="cuda"))
    W = torch.view_as_complex(torch.randn((n_rx, n_beams, 2), generator=g, device="cuda"))
    whole = rx.beamform(X, W).clone()
    for a, b in [(0, 1), (1, 2), (4, 5), (0, 2), (2, 5)]:
        assert torch.equal(rx.beamform(X[a:b].contiguous(), W), whole[a:b]), (a, b)
    rx.close()


@pytest.mark.parametrize("n_rx,n_beams,n_sc", [(48, 24, 601), (80, 24, 333)])
def test_chunk_runs_are_bit_identical_between_17_and_32_beams(n_rx, n_beams, n_sc):
    n = 5
    cell = synth.SMALL_FP32.with_(n_rx=n_rx, n_beams=n_beams, n_sc=n_sc, n_fft=1024, beam="dft")
    slots = synth.make_slots(cell, n)
    rx = host.Receiver(host.cfg_for(cell, B.PUSCH_FORM_FP32), max_slots=n)
    t, w, p = host.time_tensor(slots), host.beam_tensor(slots[0].W), host.pilot_tensor(slots)
    one = [v.clone() for v in rx.slot(t, w, p)]
    for k in (2, 3, 5):
        rx.set_pipeline(k)
        out = rx.slot(t, w, p)
        torch.cuda.synchronize()
        assert all(torch.equal(u, v) for u, v in zip(out, one)), k
    rx.close()
