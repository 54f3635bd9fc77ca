"""A destroyed handle gives back what it held, the learned estimator's workspace (40 MB here) included."""
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import denoiser as D
from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu


def test_the_learned_estimators_workspace_is_freed():
    cell = synth.DEPLOY
    params = torch.zeros(D.PARAMS, dtype=torch.bfloat16, device="cuda")
    beam = torch.ones((1, 14, cell.n_sc, cell.n_beams), dtype=torch.complex64, device="cuda")
    pilots = torch.ones((1, cell.n_layers, 2, cell.n_sc), dtype=torch.complex64, device="cuda")
    H = None

    def use():
        nonlocal H
        rx = host.Receiver(host.cfg_for(cell), max_slots=1)
        H = rx.H_buffer(1) if H is None else H
        B.pusch_chest_cnn(rx.h, 1, beam, pilots, params, 2.0, H, None, None)
        torch.cuda.synchronize()
        rx.close()

    use()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(10):
        use()
    assert free - torch.cuda.mem_get_info()[0] < 100 << 20
