"""The bench names the FP32 beamforming kernel that the library launches, on either side of every line of its choice."""
import importlib.util
from pathlib import Path

import pytest

from paper_2210_09196_gb300 import synth

ROOT = Path(__file__).resolve().parents[1]


@pytest.mark.parametrize("n_rx,n_beams,n_sc,name", [
    (64, 32, 3276, "beamform_tf32_kernel"), (256, 64, 3276, "beamform_tf32k_kernel"), (64, 33, 25, "beamform_tf32k_kernel"),
    (64, 31, 513, "beamform_tf32k_kernel"), (64, 31, 512, "beamform_fp32_kernel"), (65, 17, 25, "beamform_tf32k_kernel"),
    (32, 24, 1024, "beamform_tf32_kernel"), (32, 25, 1025, "beamform_tf32k_kernel"), (32, 25, 1023, "beamform_fp32_kernel"),
    (256, 16, 3276, "beamform_fp32_kernel"), (31, 31, 3276, "beamform_fp32_kernel"), (256, 32, 1200, "beamform_tf32k_kernel")])
def test_fp32_beamforming_kernel_name(n_rx, n_beams, n_sc, name):
    spec = importlib.util.spec_from_file_location("bench", ROOT / "bench.py")
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    cell = synth.SMALL_FP32.with_(n_rx=n_rx, n_beams=n_beams, n_sc=n_sc, n_fft=4096)
    assert b.kernel_of("beamform", "fp32", cell)[0] == name
