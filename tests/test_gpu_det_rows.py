"""The 16- and 32-lane detector (32 and 64 beams, 12 data symbols) at the edges of its warps and CTAs: one subcarrier
per slot (every subcarrier of a CTA in another slot), slot counts that leave the last warp or CTA part-filled, and layer
counts below the class, against the FP64 solve of Eq. 2 on the same estimate. Bar: 1e-5 norm-relative per slot (kappa of
these Gram matrices is below 1e3, where FP32 holds it); the decisions equal those of the detected symbols."""
import numpy as np
import pytest
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import host, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_layers,n_beams,n_sc,n", [(9, 32, 1, 7), (16, 32, 3, 3), (16, 64, 1, 1), (13, 32, 129, 2),
                                                     (17, 32, 1, 5), (31, 64, 2, 3), (32, 64, 67, 1)], ids=lambda v: str(v))
def test_part_filled_warps(n_layers, n_beams, n_sc, n):
    rng = np.random.default_rng(n_layers * 100 + n_sc)
    cfg = B.make_cfg(n_rx=n_beams, n_fft=256, n_sc=n_sc, n_beams=n_beams, n_layers=n_layers, comb=1, ports=[0] * n_layers,
                     qam_bits=4, noise_var=0.05)
    rx = host.Receiver(cfg, max_slots=n)
    H = ((rng.standard_normal((n, n_sc, n_layers, n_beams)) + 1j * rng.standard_normal((n, n_sc, n_layers, n_beams)))
         / np.sqrt(2)).astype(np.complex64)
    Y = (rng.standard_normal((n, 14, n_sc, n_beams)) + 1j * rng.standard_normal((n, 14, n_sc, n_beams))).astype(np.complex64)
    x, bits, st = rx.mmse_detect(torch.from_numpy(H).cuda(), torch.from_numpy(Y).cuda())
    torch.cuda.synchronize()
    xg = x.cpu().numpy()
    assert st.cpu().numpy()[0] == 0
    Hd = H.astype(np.complex128)
    G = np.matmul(Hd.conj(), Hd.transpose(0, 1, 3, 2)) + np.float32(0.05) * np.eye(n_layers)
    r = np.matmul(Hd.conj(), Y[:, list(synth.DATA_SYMBOLS)].astype(np.complex128).transpose(0, 2, 3, 1))
    ref = np.linalg.solve(G, r).transpose(0, 2, 3, 1)
    for i in range(n):
        assert np.linalg.norm(xg[i] - ref[i]) < 1e-5 * np.linalg.norm(ref[i])
    thr = np.float32(2 / np.sqrt(10))
    want = ((xg.real < 0).astype(np.uint8) | ((xg.imag < 0).astype(np.uint8) << 1)
            | ((np.abs(xg.real) > thr).astype(np.uint8) << 2) | ((np.abs(xg.imag) > thr).astype(np.uint8) << 3))
    assert np.array_equal(bits.cpu().numpy(), want)
    rx.close()
