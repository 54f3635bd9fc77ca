"""pusch_ls_grid (the learned estimator's input): LS values at the pilots of both DMRS symbols, interpolated over the
subcarriers, scaled by their RMS and rounded to BF16.

Widths and combs where the pilots end inside, at and before the last subcarrier, one pilot per layer, and more
pilots than shared memory holds (comb 1). Against 64 bits: BF16 rounds by at most 2^-9 of the value, the FP32
arithmetic adds about 1e-6 of the RMS."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sc,n_layers", [(300, 4), (301, 4), (257, 16), (8, 8), (9, 8), (3276, 2), (1201, 1), (3276, 1)])
def test_ls_grid_against_64_bits(n_sc, n_layers):
    n_b, n_slots = max(8, n_layers), 2
    cfg = B.make_cfg(n_rx=8, n_fft=4096, n_sc=n_sc, n_beams=n_b, n_layers=n_layers, comb=n_layers,
                     ports=list(range(n_layers)), qam_bits=2, noise_var=0.01, form=B.PUSCH_FORM_FP32)
    rx = host.Receiver(cfg, max_slots=n_slots)
    rng = np.random.default_rng(n_sc + n_layers)
    c = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)).astype(np.complex64)
    beam, pilots = c(n_slots, 14, n_sc, n_b), c(n_slots, n_layers, 2, n_sc) + 3
    grid = torch.empty((n_slots, n_layers, n_b, 2, 2, n_sc), dtype=torch.bfloat16, device="cuda")
    scale = torch.empty((n_slots, n_layers, n_b), dtype=torch.float32, device="cuda")
    B.pusch_ls_grid(rx.h, n_slots, torch.from_numpy(beam).cuda(), torch.from_numpy(pilots).cuda(), grid, scale)
    torch.cuda.synchronize()
    got, sc = grid.float().cpu().numpy().astype(np.float64), scale.cpu().numpy().astype(np.float64)
    a = np.arange(n_sc)
    for s in range(n_slots):
        for l in range(n_layers):
            q = np.arange(l, n_sc, n_layers)
            v = []
            for j, sym in enumerate((int(cfg.dmrs_sym[0]), int(cfg.dmrs_sym[1]))):
                ls = beam[s, sym, q].astype(np.complex128) / pilots[s, l, j, q].astype(np.complex128)[:, None]
                v.append(np.stack([np.interp(a, q, ls[:, b].real) + 1j * np.interp(a, q, ls[:, b].imag)
                                   for b in range(n_b)]))
            v = np.stack(v, axis=1)                                     # [B][2][n_sc]
            rms = np.sqrt(np.mean(np.abs(v) ** 2, axis=(1, 2)))
            assert np.allclose(sc[s, l], rms, rtol=1e-5)
            ref = np.stack([v.real, v.imag], axis=1) / rms[:, None, None, None]
            assert np.all(np.abs(got[s, l] - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4)
    rx.close()
