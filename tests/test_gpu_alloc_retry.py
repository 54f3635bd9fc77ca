"""A call that could not allocate all of its workspace leaves none of it behind: made again when there is memory, it gives what
a fresh handle gives. The workspaces are allocated on first use, for all slots of the handle, so the memory is taken up
between the creation of the handle and that call, down to what holds the first buffers but not all (the kernels have
run before, on another handle)."""
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import denoiser as D
from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu

SLOTS = 32
MIB = 1 << 20


def leave(mib):
    """A tensor that takes up all device memory but about `mib`."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - mib * MIB, dtype=torch.uint8, device="cuda")


def test_learned_estimator_after_a_failed_allocation():
    cell = synth.DEPLOY
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    params = torch.from_numpy(D.init_params(1)).cuda().to(torch.bfloat16)
    beam = torch.view_as_complex(torch.randn((1, 14, cell.n_sc, cell.n_beams, 2), generator=g, device="cuda"))
    pilots = torch.view_as_complex(torch.randn((1, cell.n_layers, 2, cell.n_sc, 2), generator=g, device="cuda"))
    rx = host.Receiver(host.cfg_for(cell), max_slots=1)
    want, H = rx.H_buffer(1), rx.H_buffer(1)
    B.pusch_chest_cnn(rx.h, 1, beam, pilots, params, 2.0, want, None, None)
    torch.cuda.synchronize()
    rx.close()
    rx = host.Receiver(host.cfg_for(cell), max_slots=SLOTS)
    filler = leave(700)                                   # grids 410 MiB, then 820 MiB of outputs
    with pytest.raises(B.PuschError) as ei:
        B.pusch_chest_cnn(rx.h, 1, beam, pilots, params, 2.0, H, None, None)
    assert ei.value.code == B.PUSCH_ERR_CUDA
    assert torch.cuda.mem_get_info()[0] > 600 * MIB       # nothing kept
    del filler
    torch.cuda.empty_cache()
    B.pusch_chest_cnn(rx.h, 1, beam, pilots, params, 2.0, H, None, None)
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(H), torch.view_as_real(want))
    rx.close()


def test_host_buffers_after_a_failed_allocation():
    cell = synth.DEPLOY.with_(n_rx=64, n_sc=3276)
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    t = (torch.randn((1, 14, cell.n_rx, 4096, 2), generator=g, device="cuda") * 0.02).half().cpu().pin_memory()
    p = torch.view_as_complex(torch.randn((1, cell.n_layers, 2, cell.n_sc, 2), generator=g, device="cuda")).cpu().pin_memory()
    w = torch.view_as_complex(torch.randn((cell.n_rx, cell.n_beams, 2), generator=g, device="cuda"))

    def outputs(rx):
        return (rx.xhat_buffer(1, "cpu").pin_memory(), rx.bits_buffer(1, "cpu").pin_memory(),
                rx.status_buffer("cpu").pin_memory())

    cfg = host.cfg_for(cell, B.PUSCH_FORM_MIXED)
    rx = host.Receiver(cfg, max_slots=1)
    want = outputs(rx)
    rx.slot_host(t, w, p, want)
    rx.close()
    rx = host.Receiver(cfg, max_slots=SLOTS)
    out = outputs(rx)
    filler = leave(600)                                   # samples 448 MiB, pilots 26, then 154 MiB of symbols
    with pytest.raises(B.PuschError) as ei:
        rx.slot_host(t, w, p, out)
    assert ei.value.code == B.PUSCH_ERR_CUDA
    assert torch.cuda.mem_get_info()[0] > 500 * MIB
    del filler
    torch.cuda.empty_cache()
    rx.slot_host(t, w, p, out)
    for u, v in zip(out, want):
        assert torch.equal(torch.view_as_real(u) if u.is_complex() else u, torch.view_as_real(v) if v.is_complex() else v)
    rx.close()
