"""Timed calls of the PUSCH receive path: what a receiver program runs, through the package's public entry points.

Kinds of call
  slot    the whole chain on time samples (Receiver.slot)
  fft     OFDM demodulation alone (Receiver.ofdm_fft)
  bf      beamforming alone, on an FFT output in the form's layout (Receiver.beamform)
  detect  estimation and detection on a beamformed grid: LS estimate, noise estimate if asked for, MMSE detection
  batch   a ragged multi-cell batch (RaggedReceiver.run)
  cnn     the learned estimator on a beamformed grid (pusch_chest_cnn), with the committed weights
  train   one training step of the learned estimator: forward, backward, Adam

Inputs are synthetic and made on the GPU from the seed: multipath channels of a 30 ns delay spread (the low end of
the generator's 30..1000 ns), unit-energy QPSK or 16-QAM, white noise at the case's SNR, comb or type-1 pilots. At
this delay spread the linear interpolation between pilots is accurate, so hard decisions are taken well away from
their thresholds, as they are in a link that works.
"""
import math
import os
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2210_09196_gb300 import binding as B
from paper_2210_09196_gb300 import denoiser as D
from paper_2210_09196_gb300 import host, synth

_DMRS = synth.DMRS_SYMBOLS
_DATA = synth.DATA_SYMBOLS
_FORM = {"fp32": B.PUSCH_FORM_FP32, "mixed": B.PUSCH_FORM_MIXED, "fp8": B.PUSCH_FORM_FP8}
_TAPS, _TAP_S, _SPREAD_S = 8, 15e-9, 30e-9
_SYM_S = (1.0 + 0.0703125) / 30e3
_WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(B.__file__)), "denoiser_c4.pt")


def _slot(name, **kw):
    c = dict(kind="slot", form="mixed", n_slots=1, n_rx=64, n_fft=4096, n_sc=3276, n_beams=32, n_layers=16, qam_bits=4,
             fp16=True, snr_db=30.0, pipeline=1, cp=False, shift=False, type1=False, est_noise=False, chol_every=0,
             doppler_hz=0.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one slot of the small cell, FP32: the smallest call, a receiver that decodes each slot as it arrives
        _slot("slot_small", form="fp32", n_rx=16, n_fft=512, n_sc=300, n_beams=16, n_layers=4, qam_bits=2, fp16=False,
              snr_db=20.0),
        # the deployment cell, mixed form, 16 slots a call over two streams: throughput of a loaded base station
        _slot("slot_deploy", n_slots=16, pipeline=2),
        # a standard slot with everything switched on: cyclic prefixes, type-1 pilots, estimated noise, a channel that
        # changes over the slot and one factorisation per 4 symbols
        _slot("slot_nr", n_slots=4, n_layers=4, cp=True, type1=True, est_noise=True, chol_every=4, doppler_hz=100.0),
        # the mixed form's FFT on the deployment cell, for a program that runs the stages itself
        dict(name="fft_mixed", kind="fft", form="mixed", n_slots=8, n_rx=64, n_fft=4096, n_sc=3276, fp16=True, cp=False,
             shift=False),
        # the FP8 form's FFT with block-scaled output on the massive-MIMO cell
        dict(name="fft_fp8", kind="fft", form="fp8", n_slots=2, n_rx=256, n_fft=4096, n_sc=3276, fp16=True, cp=False,
             shift=False),
        # beamforming of the massive-MIMO cell (256 antennas to 64 beams) in each of the three forms
        dict(name="bf_mixed", kind="bf", form="mixed", n_slots=4, n_rx=256, n_fft=4096, n_sc=3276, n_beams=64),
        dict(name="bf_fp8", kind="bf", form="fp8", n_slots=4, n_rx=256, n_fft=4096, n_sc=3276, n_beams=64),
        dict(name="bf_fp32", kind="bf", form="fp32", n_slots=2, n_rx=256, n_fft=4096, n_sc=3276, n_beams=64),
        # estimation and detection of the massive-MIMO cell's 32 users
        dict(name="detect_massive", kind="detect", n_slots=2, n_sc=3276, n_beams=64, n_layers=32, qam_bits=4,
             snr_db=25.0, est_noise=False),
        # 8 cells of different sizes with 64 users on their own subcarrier ranges, one graph launch a slot
        dict(name="batch_ragged", kind="batch", n_cells=8, n_users=64, layout=3),
        # the learned estimator on one slot of the deployment cell: 512 grids of 3276 subcarriers
        dict(name="cnn_estimate", kind="cnn", n_slots=1, n_sc=3276, n_beams=32, n_layers=16, snr_db=20.0),
        # its training step: 4 slot crops of 16 layers x 16 beams, 256 subcarriers each
        dict(name="cnn_train", kind="train", n_grids=1024, width=256),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_sc(rng, n_fft):
    return rng.randint(n_fft // 2, int(0.8 * n_fft))


def draw(rng):
    kind = rng.choice(["slot", "slot", "slot", "fft", "fft", "bf", "bf", "bf", "detect", "batch", "cnn", "train"])
    if kind == "slot":
        form = rng.choice(["fp32", "mixed", "mixed"])
        n_fft = rng.choice([512, 1024, 2048, 4096])
        n_beams = rng.choice([8, 16, 24, 32])
        type1 = rng.random() < 0.3
        n_layers = rng.randint(1, 4) if type1 else rng.randint(1, max(1, n_beams // 2))
        n_rx = rng.randint(n_beams, 64) if form == "fp32" else 8 * rng.randint(n_beams // 8, 8)
        n_sc = _draw_sc(rng, n_fft)
        if type1:
            n_sc &= ~3
        n_slots = _log_int(rng, 1, 16)
        return _slot(None, form=form, n_slots=n_slots, n_rx=n_rx, n_fft=n_fft, n_sc=n_sc, n_beams=n_beams,
                     n_layers=n_layers, qam_bits=rng.choice([2, 4]), fp16=form != "fp32" or rng.random() < 0.5,
                     pipeline=rng.choice([1, 2]) if n_slots > 1 else 1, cp=rng.random() < 0.3,
                     shift=rng.random() < 0.2, type1=type1, est_noise=rng.random() < 0.3,
                     chol_every=rng.choice([0, 0, 0, 4, 12]))
    if kind == "fft":
        form = rng.choice(["mixed", "mixed", "fp8", "fp32"])
        n_fft = rng.choice([512, 1024, 2048, 4096, 4096])
        n_rx = 16 * _log_int(rng, 1, 16)
        return dict(kind="fft", form=form, n_slots=rng.randint(1, max(1, 512 // n_rx)), n_rx=n_rx, n_fft=n_fft,
                    n_sc=_draw_sc(rng, n_fft), fp16=rng.random() < 0.7, cp=rng.random() < 0.3,
                    shift=rng.random() < 0.2)
    if kind == "bf":
        form = rng.choice(["mixed", "fp8", "fp32"])
        n_rx = 16 * _log_int(rng, 1, 16)
        n_fft = rng.choice([1024, 2048, 4096])
        return dict(kind="bf", form=form, n_slots=rng.randint(1, max(1, 512 // n_rx)), n_rx=n_rx, n_fft=n_fft,
                    n_sc=_draw_sc(rng, n_fft), n_beams=rng.choice([8, 16, 32, 40, 64]))
    if kind == "detect":
        n_beams = rng.choice([8, 16, 24, 32, 64])
        return dict(kind="detect", n_slots=_log_int(rng, 1, 4), n_sc=rng.randint(300, 3276), n_beams=n_beams,
                    n_layers=rng.randint(2, max(2, n_beams // 2)), qam_bits=rng.choice([2, 4]), snr_db=25.0,
                    est_noise=rng.random() < 0.5)
    if kind == "batch":
        n_cells = rng.randint(2, 8)
        return dict(kind="batch", n_cells=n_cells, n_users=rng.randint(4 * n_cells, 8 * n_cells),
                    layout=rng.randrange(1 << 20))
    if kind == "cnn":
        return dict(kind="cnn", n_slots=1, n_sc=rng.randint(600, 3276), n_beams=rng.choice([8, 16, 32]),
                    n_layers=rng.randint(2, 8), snr_db=20.0)
    return dict(kind="train", n_grids=_log_int(rng, 64, 1024), width=rng.choice([8 * rng.randint(12, 32), rng.randint(96, 256)]))


# ------------------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2 + 1)
    return g


def _cn(g, shape):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device="cuda") * math.sqrt(0.5))


def _qam(g, shape, qam_bits):
    """Unit-energy QPSK or 16-QAM symbols."""
    s = 1.0 - 2.0 * torch.randint(0, 2, tuple(shape) + (2,), generator=g, device="cuda").float()
    if qam_bits == 4:
        s = s * (1.0 + 2.0 * torch.randint(0, 2, s.shape, generator=g, device="cuda").float()) / math.sqrt(5.0)
    return torch.view_as_complex(s * math.sqrt(0.5))


def _channel(g, n_rx, n_layers, n_sc, n_fft, first=0):
    """Taps [R, L, T] and the response of each tap at the subcarriers [n_sc, T]."""
    i = torch.arange(_TAPS, device="cuda", dtype=torch.float64)
    p = torch.exp(-i * _TAP_S / _SPREAD_S)
    k = torch.arange(n_sc, device="cuda", dtype=torch.float64) + first
    F = torch.polar(torch.ones((n_sc, _TAPS), device="cuda", dtype=torch.float64),
                    -2 * math.pi * 30e3 * _TAP_S * k[:, None] * i[None, :])
    return _cn(g, (n_rx, n_layers, _TAPS)) * torch.sqrt(p / p.sum()).float(), F.to(torch.complex64)


def _comb_pilots(g, n_layers, n_sc):
    a = torch.arange(n_sc, device="cuda")
    mask = (a[None, :] % n_layers) == torch.arange(n_layers, device="cuda")[:, None]
    return _qam(g, (n_layers, 2, n_sc), 2) * mask[:, None, :]


def _grid(g, n_layers, n_sc, qam_bits, pilots):
    """Transmitted grid [L, 14, n_sc]."""
    t = torch.empty((n_layers, synth.N_SYM, n_sc), dtype=torch.complex64, device="cuda")
    t[:, list(_DATA)] = _qam(g, (n_layers, len(_DATA), n_sc), qam_bits)
    t[:, list(_DMRS)] = pilots
    return t


def _receive(g, taps, F, t, doppler_hz=0.0):
    """Noiseless received grid [14, R, n_sc]."""
    R, L, T = taps.shape
    tt = t.permute(2, 0, 1).contiguous()                                              # [n_sc, L, 14]
    if doppler_hz == 0.0:
        H = (taps.reshape(R * L, T) @ F.T).reshape(R, L, -1).permute(2, 0, 1)         # [n_sc, R, L]
        return (H @ tt).permute(2, 1, 0)
    fd = doppler_hz * torch.cos(2 * math.pi * torch.rand((R, L, T), generator=g, device="cuda"))
    out = []
    for s in range(synth.N_SYM):
        tap = taps * torch.polar(torch.ones_like(fd), 2 * math.pi * _SYM_S * s * fd)
        H = (tap.reshape(R * L, T) @ F.T).reshape(R, L, -1).permute(2, 0, 1)
        out.append((H @ tt[:, :, s:s + 1])[..., 0].T)
    return torch.stack(out)


def _waveform(X, n_fft, cp, shift, fp16):
    """Received grid [14, R, n_sc] -> time samples of one slot in the call's layout."""
    S, R, n_sc = X.shape
    spec = torch.zeros((S, R, n_fft), dtype=torch.complex64, device="cuda")
    spec[:, :, (torch.arange(n_sc, device="cuda") - n_sc // 2) % n_fft] = X
    x = torch.fft.ifft(spec, dim=-1)
    if cp or shift:
        parts = []
        for s in range(S):
            c = synth.cp_lengths(n_fft)[0 if s == 0 else 1] if cp else 0
            n = torch.arange(-c, n_fft, device="cuda")
            v = x[s][:, n % n_fft]
            if shift:
                v = v * torch.polar(torch.ones(n.numel(), device="cuda", dtype=torch.float64),
                                    2 * math.pi * n.double() / (4 * n_fft)).to(torch.complex64)
            parts.append(v)
        x = torch.cat(parts, dim=1) if cp else torch.stack(parts)
    x = x.contiguous()
    return torch.view_as_real(x).half() if fp16 else x


def _dft_beams(n_rx, n_beams):
    r = np.arange(n_rx)[:, None] * np.arange(n_beams)[None, :]
    return torch.from_numpy((np.exp(-2j * np.pi * r / n_rx) / np.sqrt(n_rx)).astype(np.complex64)).cuda()


def _cfg(c, **kw):
    a = dict(n_rx=c.get("n_rx", 16), n_fft=c.get("n_fft", 4096), n_sc=c["n_sc"], n_beams=c.get("n_beams", 8),
             n_layers=c.get("n_layers", 1), qam_bits=c.get("qam_bits", 2), in_fp16=c.get("fp16", False),
             form=_FORM[c.get("form", "fp32")], noise_var=10.0 ** (-c.get("snr_db", 30.0) / 10.0),
             chol_every=c.get("chol_every", 0), cp=c.get("cp", False), shift_7p5khz=c.get("shift", False),
             dmrs_type=1 if c.get("type1") else 0)
    if c.get("est_noise"):
        a["noise_var"] = B.PUSCH_NOISE_ESTIMATE
    a.update(kw)
    return B.make_cfg(**a)


def _slot_inputs(c, seed):
    g = _gen(seed)
    L, n_sc = c["n_layers"], c["n_sc"]
    nv = 10.0 ** (-c["snr_db"] / 10.0)
    cfg = _cfg(c)
    if c["type1"]:
        pil = torch.zeros((c["n_slots"], L, 2, n_sc), dtype=torch.complex64, device="cuda")
        B.pusch_dmrs_type1_pilots(cfg, c["n_slots"], [(seed + i) % 160 for i in range(c["n_slots"])], seed % 1008, 0, pil)
    else:
        pil = torch.stack([_comb_pilots(g, L, n_sc) for _ in range(c["n_slots"])])
    time = []
    for i in range(c["n_slots"]):
        taps, F = _channel(g, c["n_rx"], L, n_sc, c["n_fft"])
        X = _receive(g, taps, F, _grid(g, L, n_sc, c["qam_bits"], pil[i]), c["doppler_hz"])
        X = X + _cn(g, X.shape) * math.sqrt(nv)
        time.append(_waveform(X, c["n_fft"], c["cp"], c["shift"], c["fp16"]))
    return cfg, torch.stack(time), _dft_beams(c["n_rx"], c["n_beams"]), pil.contiguous()


def _fft_inputs(c, seed):
    g = _gen(seed)
    return torch.stack([_waveform(_cn(g, (synth.N_SYM, c["n_rx"], c["n_sc"])) * 4.0, c["n_fft"], c["cp"], c["shift"],
                                  c["fp16"]) for _ in range(c["n_slots"])])


def _pow2_scale(amax):
    """The smallest 2^e (e >= -126) with amax <= 448 * 2^e."""
    e = torch.ceil(torch.log2(amax.double() / 448.0))
    e = torch.where(amax.double() > 448.0 * torch.exp2(e), e + 1, e)
    e = torch.where(amax.double() <= 448.0 * torch.exp2(e - 1), e - 1, e)
    return torch.exp2(e.clamp(min=-126)).float()


def _bf_inputs(c, seed):
    """(freq buffer in the form's layout, its values as two real planes [n, 14, R, n_sc] in FP32)."""
    g = _gen(seed)
    n, R, n_sc = c["n_slots"], c["n_rx"], c["n_sc"]
    x = torch.randn((n, synth.N_SYM, R, 2, n_sc), generator=g, device="cuda") * 3.0
    if c["form"] == "fp32":
        return torch.view_as_complex(x.movedim(3, -1).contiguous()), x
    cfg = _cfg(c)
    pitch = B.pusch_sc_pitch(cfg)
    planes = torch.zeros((n, synth.N_SYM, R, 2, pitch), device="cuda")
    planes[..., :n_sc] = x
    if c["form"] == "mixed":
        q = planes.half()
        return q, q[..., :n_sc].float()
    blocks = planes.reshape(n, synth.N_SYM, R, 2, pitch // 128, 128)
    scale = _pow2_scale(blocks.abs().amax(dim=(3, 5)).clamp(min=1e-30))                # [n, 14, R, blk]
    codes = (blocks / scale[:, :, :, None, :, None]).to(torch.float8_e4m3fn)
    val = (codes.float() * scale[:, :, :, None, :, None]).reshape(planes.shape)[..., :n_sc]
    buf = torch.zeros(B.pusch_freq_bytes(cfg, n), dtype=torch.uint8, device="cuda")
    buf[:codes.numel()] = codes.reshape(-1).view(torch.uint8)
    sc = scale.permute(0, 1, 3, 2).contiguous().reshape(-1).view(torch.uint8)          # [n, 14, blk, R]
    buf[buf.numel() - sc.numel():] = sc
    return buf, val


def _detect_inputs(c, seed):
    """Beamformed grid [n, 14, n_sc, B] and pilots [n, L, 2, n_sc]."""
    g = _gen(seed)
    nv = 10.0 ** (-c["snr_db"] / 10.0)
    pil, beam = [], []
    for _ in range(c["n_slots"]):
        p = _comb_pilots(g, c["n_layers"], c["n_sc"])
        taps, F = _channel(g, c["n_beams"], c["n_layers"], c["n_sc"], 4096)
        X = _receive(g, taps, F, _grid(g, c["n_layers"], c["n_sc"], c.get("qam_bits", 4), p))
        X = X + _cn(g, X.shape) * math.sqrt(nv)
        pil.append(p)
        beam.append(X.transpose(1, 2).contiguous())
    return torch.stack(beam), torch.stack(pil)


def _layout(c):
    """Cells and users of a ragged batch: 32 or 64 antennas, 2048- or 4096-point FFTs, a user on a contiguous range of
    resource blocks with the lowest ports that no overlapping user has, at most n_beams / 2 layers on a subcarrier."""
    rng = random.Random(c["layout"])
    cells, users = [], []
    for _ in range(c["n_cells"]):
        n_rx, n_fft = rng.choice([32, 64]), rng.choice([2048, 4096])
        cells.append(synth.RaggedCell(n_rx=n_rx, n_fft=n_fft, n_sc=12 * int(0.8 * n_fft / 12), n_beams=n_rx // 2,
                                      noise_var=10.0 ** -2.5, comb=n_rx // 4))
    placed = [[] for _ in cells]
    for _ in range(50 * c["n_users"]):                  # a layout too full for more users has fewer
        if len(users) == c["n_users"]:
            break
        k = rng.randrange(len(cells))
        cell = cells[k]
        prbs = cell.n_sc // 12
        n_prb = rng.randint(4, prbs)
        a0 = 12 * rng.randint(0, prbs - n_prb)
        a1, L = a0 + 12 * n_prb, rng.randint(1, 4)
        near = [u for u in placed[k] if u[0] < a1 and a0 < u[1]]
        free = [p for p in range(cell.comb - L + 1) if all(p + L <= q or q + m <= p for _, _, q, m in near)]
        if not free:
            continue
        placed[k].append((a0, a1, free[0], L))
        users.append(synth.RaggedUser(cell=k, sc_start=a0, sc_count=a1 - a0, n_layers=L, port0=free[0],
                                      qam_bits=rng.choice([2, 4]), snr_db=rng.uniform(20.0, 25.0)))
    return cells, users


def _batch_inputs(c, seed):
    g = _gen(seed)
    cells, users = _layout(c)
    X = [_cn(g, (synth.N_SYM, k.n_rx, k.n_sc)) * math.sqrt(k.noise_var) for k in cells]
    pil = []
    for u in users:
        k = cells[u.cell]
        a = torch.arange(u.sc_start, u.sc_start + u.sc_count, device="cuda")
        mask = (a[None, :] % k.comb) == (u.port0 + torch.arange(u.n_layers, device="cuda"))[:, None]
        p = _qam(g, (u.n_layers, 2, u.sc_count), 2) * mask[:, None, :]
        taps, F = _channel(g, k.n_rx, u.n_layers, u.sc_count, k.n_fft, u.sc_start)
        gain = math.sqrt(10.0 ** (u.snr_db / 10.0) * k.noise_var)
        X[u.cell][:, :, u.sc_start:u.sc_start + u.sc_count] += gain * _receive(
            g, taps, F, _grid(g, u.n_layers, u.sc_count, u.qam_bits, p))
        pil.append(p.reshape(-1))
    time = [_waveform(X[i], k.n_fft, False, False, True) for i, k in enumerate(cells)]
    return (cells, users, torch.cat([t.reshape(-1, 2) for t in time]),
            torch.cat([_dft_beams(k.n_rx, k.n_beams).reshape(-1) for k in cells]), torch.cat(pil), time)


def _train_inputs(c, seed):
    """Training data and a trainer's state some way into a run (parameters, moments)."""
    g = _gen(seed)
    n, w = c["n_grids"], c["width"]
    p = torch.from_numpy(D.init_params(seed % 1000)).cuda()
    p = p + 0.01 * torch.randn(p.shape, generator=g, device="cuda")
    target = torch.randn((n, 2, 2, w), generator=g, device="cuda")
    target = torch.nn.functional.avg_pool1d(target.reshape(n * 4, 1, w), 9, 1, 4, count_include_pad=False)
    target = (target / target.std()).reshape(n, 2, 2, w).contiguous()
    x = (target + 0.3 * torch.randn(target.shape, generator=g, device="cuda")).to(torch.bfloat16)
    m = 1e-3 * torch.randn(p.shape, generator=g, device="cuda")
    v = 1e-5 * (0.1 + torch.rand(p.shape, generator=g, device="cuda"))
    return x, target, p, m, v


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = SimpleNamespace(case=c)
    if kind == "slot":
        cfg, s.time, s.W, s.pilots = _slot_inputs(c, seed)
        s.rx = host.Receiver(cfg, max_slots=c["n_slots"])
        if c["pipeline"] > 1:
            s.rx.set_pipeline(c["pipeline"])
        s.out = (s.rx.xhat_buffer(c["n_slots"]), s.rx.bits_buffer(c["n_slots"]), s.rx.status_buffer())
    elif kind == "fft":
        s.time = _fft_inputs(c, seed)
        s.rx = host.Receiver(_cfg(c), max_slots=c["n_slots"])
        s.freq = s.rx.freq_buffer(c["n_slots"]).zero_()
    elif kind == "bf":
        s.freq, _ = _bf_inputs(c, seed)
        s.W = _dft_beams(c["n_rx"], c["n_beams"])
        s.rx = host.Receiver(_cfg(c), max_slots=c["n_slots"])
        s.beam = s.rx.beam_buffer(c["n_slots"])
    elif kind == "detect":
        s.beam, s.pilots = _detect_inputs(c, seed)
        s.rx = host.Receiver(_cfg(c, n_rx=c["n_beams"]), max_slots=c["n_slots"])
        s.H = s.rx.H_buffer(c["n_slots"])
    elif kind == "batch":
        cells, users, s.time, s.W, s.pilots, _ = _batch_inputs(c, seed)
        s.rx = host.RaggedReceiver(SimpleNamespace(cells=cells, users=users), B.PUSCH_FORM_MIXED)
        s.out = s.rx.outputs()
    elif kind == "cnn":
        s.beam, s.pilots = _detect_inputs(c, seed)
        s.params, _ = D.load_weights(_WEIGHTS)
        s.rx = host.Receiver(_cfg(c, n_rx=c["n_beams"]), max_slots=c["n_slots"])
        s.H = s.rx.H_buffer(c["n_slots"])
        grids = c["n_slots"] * c["n_layers"] * c["n_beams"]
        s.resid = torch.zeros(grids, device="cuda")
        s.fallback = torch.zeros(grids, dtype=torch.uint8, device="cuda")
    else:
        n, w = c["n_grids"], c["width"]
        s.x, s.target, s.p0, s.m0, s.v0 = _train_inputs(c, seed)
        s.p, s.m, s.v = s.p0.clone(), s.m0.clone(), s.v0.clone()
        s.pb = s.p.to(torch.bfloat16)
        s.grad = torch.zeros_like(s.p)
        s.y = torch.zeros((n, 2, 2, w), device="cuda")
        s.acts = torch.zeros((3, n, 32, 2, w), dtype=torch.bfloat16, device="cuda")
        s.work = torch.zeros(2 * n * 32 * 2 * w, device="cuda")
        s.wflip = torch.zeros(D.PARAMS, dtype=torch.bfloat16, device="cuda")
        s.loss = torch.zeros(1, device="cuda")
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "slot":
        x, bits, status = s.rx.slot(s.time, s.W, s.pilots, s.out)
        return {"x_hat": x, "bits": bits, "status": status}
    if kind == "fft":
        f = s.rx.ofdm_fft(s.time, s.freq)
        if c["form"] != "fp8":
            return {"freq": f}
        rows = c["n_slots"] * synth.N_SYM * c["n_rx"]
        scales = rows * -(-c["n_sc"] // 128)
        return {"codes": f[:rows * 2 * s.rx.pitch].view(torch.float8_e4m3fn),
                "scales": f[f.numel() - 4 * scales:].view(torch.float32)}
    if kind == "bf":
        return {"beam": s.rx.beamform(s.freq, s.W, s.beam)}
    if kind == "detect":
        out = {"H": s.rx.chest_ls(s.beam, s.pilots, s.H)}
        if c["est_noise"]:
            out["sigma2"] = s.rx.noise_estimate(s.beam, s.pilots)
        out["x_hat"], out["bits"], out["status"] = s.rx.mmse_detect(s.H, s.beam)
        return out
    if kind == "batch":
        x, bits, status = s.rx.run(s.time, s.W, s.pilots, s.out)
        return {"x_hat": x, "bits": bits, "status": status}
    if kind == "cnn":
        B.pusch_chest_cnn(s.rx.h, c["n_slots"], s.beam, s.pilots, s.params, 2.0, s.H, s.resid, s.fallback)
        return {"H": s.H, "resid": s.resid, "fallback": s.fallback}
    # a training step from the same parameters and moments on every pass
    n, w = c["n_grids"], c["width"]
    s.p.copy_(s.p0)
    s.m.copy_(s.m0)
    s.v.copy_(s.v0)
    s.pb.copy_(s.p0)
    B.pusch_cnn_forward(n, w, s.x, s.pb, s.y, s.acts)
    B.pusch_cnn_backward(n, w, s.x, s.acts, s.pb, s.y, s.target, s.grad, s.loss, s.work, s.wflip)
    B.pusch_cnn_adam(200, 1e-3, 0.9, 0.999, 1e-8, s.p, s.pb, s.grad, s.m, s.v)
    return {"y": s.y, "acts": s.acts, "loss": s.loss, "grad": s.grad, "p": s.p, "pb": s.pb, "m": s.m, "v": s.v}


# ---------------------------------------------------------------------------------------------------------- the work
def _det_flops(n_sc, L, Bm, groups):
    cmac = groups * (L * (L + 1) / 2 * Bm + L ** 3 / 6) + 12 * L * Bm + 12 * L * L
    return 8.0 * n_sc * cmac


def work(case):
    c, kind, S = case, case["kind"], synth.N_SYM
    if kind == "batch":
        cells, users = _layout(c)
        by = sum(S * k.n_rx * k.n_fft * 4 + k.n_rx * k.n_beams * 8 for k in cells)
        fl = sum(S * k.n_rx * 5 * k.n_fft * math.log2(k.n_fft) + 8.0 * S * k.n_sc * k.n_rx * k.n_beams for k in cells)
        active = [np.zeros(k.n_sc, dtype=int) for k in cells]
        for u in users:
            k = cells[u.cell]
            by += u.n_layers * (2 * 8 * u.sc_count / k.comb + 12 * u.sc_count * 9)
            active[u.cell][u.sc_start:u.sc_start + u.sc_count] += u.n_layers
        for k, a in zip(cells, active):
            fl += sum(_det_flops(int((a == L).sum()), int(L), k.n_beams, 1) for L in set(a.tolist()) if L)
        return {"bytes": by, "flops": fl}
    if kind == "train":
        n, w = c["n_grids"], c["width"]
        pixels = n * 2 * w
        by = pixels * (2 * 2 + 2 * 4 + 2 * 4 + 96 * 2) + D.PARAMS * (4 * 7 + 2)
        return {"bytes": by, "flops": 2.0 * pixels * (2.0 / 3.0) * (3 * 19584 - 576)}
    n, n_sc, R, Bm, L = c["n_slots"], c["n_sc"], c.get("n_rx", 0), c.get("n_beams", 0), c.get("n_layers", 0)
    form = c.get("form", "fp32")
    value = {"fp32": 8, "mixed": 4, "fp8": 2}[form]
    samples = 0
    if kind in ("slot", "fft"):
        samples = S * R * c["n_fft"] * (4 if c["fp16"] else 8)
    fft_fl = S * R * 5.0 * c.get("n_fft", 2) * math.log2(c.get("n_fft", 2))
    if kind == "fft":
        return {"bytes": n * (samples + S * R * n_sc * value), "flops": n * fft_fl}
    if kind == "bf":
        return {"bytes": n * S * n_sc * (R * value + Bm * 8) + R * Bm * 8, "flops": n * 8.0 * S * n_sc * R * Bm}
    used_pilots = n_sc * 2 * 8 * (L / 2 if c.get("type1") else 1)
    out = L * 12 * n_sc * 9
    groups = -(-12 // c["chol_every"]) if c.get("chol_every") else 1
    if kind == "slot":
        return {"bytes": n * (samples + used_pilots + out) + R * Bm * 8,
                "flops": n * (fft_fl + 8.0 * S * n_sc * R * Bm + _det_flops(n_sc, L, Bm, groups))}
    if kind == "detect":
        return {"bytes": n * (S * n_sc * Bm * 8 + used_pilots + n_sc * L * Bm * 8 + out),
                "flops": n * _det_flops(n_sc, L, Bm, 1)}
    return {"bytes": n * (2 * n_sc * Bm * 8 + used_pilots + n_sc * L * Bm * 8) + D.PARAMS * 2,
            "flops": n * L * Bm * 2 * n_sc * 2.0 * (2.0 / 3.0) * 19584}


# ----------------------------------------------------------------------------------------- the same values in 64 bits
def _x_demod(t, n_fft, n_sc, cp, shift):
    """[.., time samples of a slot] -> [14, R, n_sc] complex128."""
    x = torch.view_as_complex(t.double()) if t.dtype == torch.float16 else t.to(torch.complex128)
    S = synth.N_SYM
    if cp:
        c0, c1 = 352 * n_fft // 4096, 288 * n_fft // 4096
        x = torch.stack([x[:, s * (n_fft + c1) + c0:s * (n_fft + c1) + c0 + n_fft] for s in range(S)])
    if shift:
        n = torch.arange(n_fft, device=x.device, dtype=torch.float64)
        x = x * torch.polar(torch.ones_like(n), -2 * math.pi * n / (4 * n_fft))
    return torch.fft.fft(x, dim=-1)[..., (torch.arange(n_sc, device=x.device) - n_sc // 2) % n_fft]


def _x_interp(v, first, step, n):
    """Values [.., K, B] at positions first + k step -> [.., n, B] by linear interpolation, held outside."""
    a = torch.arange(n, device=v.device, dtype=torch.float64)
    u = ((a - first) / step).clamp(0, v.shape[-2] - 1)
    lo = u.floor().long()
    hi = (lo + 1).clamp(max=v.shape[-2] - 1)
    w = (u - lo)[:, None]
    return v[..., lo, :] * (1 - w) + v[..., hi, :] * w


def _x_ls(Y, pil, ports, comb, type1):
    """Per-DMRS-symbol estimates [2, L, n_sc, B] from the beamformed grid [14, n_sc, B]."""
    n_sc = Y.shape[1]
    p = pil.to(torch.complex128)
    out = []
    for j, s in enumerate(_DMRS):
        rows = []
        for l, port in enumerate(ports):
            if type1:
                k = torch.arange(port // 2, n_sc, 2, device=Y.device)
                v = Y[s, k] / p[l, j, k][:, None]
                rows.append(_x_interp(0.5 * (v[0::2] + v[1::2]), port // 2 + 1, 4, n_sc))
            else:
                k = torch.arange(port, n_sc, comb, device=Y.device)
                rows.append(_x_interp(Y[s, k] / p[l, j, k][:, None], port, comb, n_sc))
        out.append(torch.stack(rows))
    return torch.stack(out)


def _x_noise(Y, pil, ports, comb, type1):
    """Noise variance from the pilot residuals of one slot."""
    n_sc = Y.shape[1]
    p = pil.to(torch.complex128)
    num, den = 0.0, 0.0
    for grp in ([0, 1] if type1 else range(len(ports))):
        ls = [l for l, q in enumerate(ports) if q // 2 == grp] if type1 else [grp]
        if not ls:
            continue
        k = torch.arange(grp if type1 else ports[grp], n_sc, 2 if type1 else comb, device=Y.device)
        y = Y[list(_DMRS)][:, k]                                                        # [2, K, B]
        if type1:
            y = y.reshape(2, -1, 2, y.shape[-1])                                        # [2, pairs, 2, B]
            q = [p[l][:, k].reshape(2, -1, 2, 1) for l in ls]
            fit = sum(0.25 * (y / v).sum(dim=(0, 2), keepdim=True) * v for v in q)
            num = num + (y - fit).abs().square().sum()
            den += y.shape[1] * y.shape[3] * (4 - len(ls))
        else:
            v = p[ls[0]][:, k][..., None]
            num = num + (y - 0.5 * (y / v).sum(0, keepdim=True) * v).abs().square().sum()
            den += y.numel() / 2
    return float(num) / den


def _x_solve(H, Y, load):
    """H [n_sc, L, B], Y [n_sym, n_sc, B] -> x [L, n_sym, n_sc] of Eq. 2."""
    Hc = H.conj()
    G = Hc @ H.transpose(1, 2)
    G = G + load * torch.eye(G.shape[-1], device=G.device, dtype=G.dtype)
    return torch.linalg.solve(G, Hc @ Y.permute(1, 2, 0)).permute(1, 2, 0)


def _x_slot(c, cfg, t, W, pil):
    X = _x_demod(t, c["n_fft"], c["n_sc"], c["cp"], c["shift"])
    Y = torch.einsum("srk,rb->skb", X, W.to(torch.complex128).conj())
    L = c["n_layers"]
    ports, comb = list(range(L)), L
    E = _x_ls(Y, pil, ports, comb, c["type1"])
    nv = _x_noise(Y, pil, ports, comb, c["type1"]) if c["est_noise"] else float(cfg.noise_var)
    data = list(_DATA)
    if not c["chol_every"]:
        return _x_solve(E.mean(0).transpose(0, 1), Y[data], nv)
    parts = []
    for d in range(0, 12, c["chol_every"]):
        sy = data[d:d + c["chol_every"]]
        u = sum((s - _DMRS[0]) / (_DMRS[1] - _DMRS[0]) for s in sy) / len(sy)
        parts.append(_x_solve((E[0] + u * (E[1] - E[0])).transpose(0, 1), Y[sy], nv))
    return torch.cat(parts, dim=1)


def _x_params(p):
    """[(W, b)] of the four layers in float64."""
    out, o, ch = [], 0, (2, 32, 32, 32, 2)
    for k in range(4):
        n = ch[k] * ch[k + 1] * 9
        out.append((p[o:o + n].reshape(ch[k + 1], ch[k], 3, 3), p[o + n:o + n + ch[k + 1]]))
        o += n + ch[k + 1]
    return out


def _x_forward(x, p):
    """(y, activations) of the denoiser; the dilated convolutions as 9 shifted products, so that they run anywhere."""
    a, acts = x, []
    for k, ((W, b), dil) in enumerate(zip(_x_params(p), (1, 8, 16, 1))):
        w = a.shape[-1]
        pad = torch.nn.functional.pad(a, (dil, dil, 1, 1))
        z = b[None, :, None, None]
        for kh in range(3):
            for kw in range(3):
                z = z + torch.einsum("oc,nchw->nohw", W[:, :, kh, kw], pad[:, :, kh:kh + 2, kw * dil:kw * dil + w])
        a = z if k == 3 else torch.relu(z)
        if k < 3:
            acts.append(a)
    return a + x, acts


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "slot":
        cfg, t, W, pil = _slot_inputs(c, seed)
        x = torch.stack([_x_slot(c, cfg, t[i], W, pil[i]) for i in range(c["n_slots"])])
        return {"x_hat": x, "bits": None, "status": None}
    if kind == "fft":
        X = torch.stack([_x_demod(t, c["n_fft"], c["n_sc"], c["cp"], c["shift"]) for t in _fft_inputs(c, seed)])
        if c["form"] == "fp32":
            return {"freq": X}
        pitch = B.pusch_sc_pitch(_cfg(c))
        P = torch.zeros(X.shape[:3] + (2, pitch), dtype=torch.float64, device="cuda")
        P[..., :c["n_sc"]] = torch.view_as_real(X).movedim(-1, 3)
        if c["form"] == "mixed":
            return {"freq": P}
        blk = P.reshape(X.shape[:3] + (2, pitch // 128, 128))
        sc = _pow2_scale(blk.abs().amax(dim=(3, 5)).clamp(min=1e-300))
        return {"codes": (blk / sc.double()[:, :, :, None, :, None]).reshape(-1),
                "scales": sc.double().permute(0, 1, 3, 2).reshape(-1)}
    if kind == "bf":
        _, val = _bf_inputs(c, seed)
        W = torch.view_as_real(_dft_beams(c["n_rx"], c["n_beams"])).double()            # [R, B, 2]
        if c["form"] == "mixed":
            W = W.half().double()
        if c["form"] == "fp8":
            for r in range(0, c["n_rx"], 128):
                s = _pow2_scale(W[r:r + 128].abs().amax(dim=(0, 2))).double()[None, :, None]
                W[r:r + 128] = (W[r:r + 128] / s).float().to(torch.float8_e4m3fn).double() * s
        W = torch.view_as_complex(W.contiguous()).conj()
        out = [torch.einsum("srk,rb->skb", torch.view_as_complex(v.movedim(2, -1).double().contiguous()), W) for v in val]
        return {"beam": torch.stack(out)}
    if kind == "detect":
        beam, pil = _detect_inputs(c, seed)
        L = c["n_layers"]
        nv = float(_cfg(c, n_rx=c["n_beams"]).noise_var)
        H, x, sig = [], [], []
        for i in range(c["n_slots"]):
            Y = beam[i].to(torch.complex128)
            H.append(_x_ls(Y, pil[i], range(L), L, False).mean(0).transpose(0, 1).contiguous())
            sig.append(_x_noise(Y, pil[i], range(L), L, False))
            x.append(_x_solve(H[-1], Y[list(_DATA)], sig[-1] if c["est_noise"] else nv))
        out = {"H": torch.stack(H), "x_hat": torch.stack(x), "bits": None, "status": None}
        if c["est_noise"]:
            out["sigma2"] = torch.tensor(sig, dtype=torch.float64, device="cuda")
        return out
    if kind == "batch":
        cells, users, _, _, _, time = _batch_inputs(c, seed)
        o, pils = 0, []
        flat = _batch_inputs(c, seed)[4]
        for u in users:
            n = u.n_layers * 2 * u.sc_count
            pils.append(flat[o:o + n].reshape(u.n_layers, 2, u.sc_count))
            o += n
        xs = [torch.zeros((u.n_layers, 12, u.sc_count), dtype=torch.complex128, device="cuda") for u in users]
        for k, cell in enumerate(cells):
            X = _x_demod(time[k], cell.n_fft, cell.n_sc, False, False)
            Y = torch.einsum("srk,rb->skb", X, _dft_beams(cell.n_rx, cell.n_beams).to(torch.complex128).conj())
            mine = [i for i, u in enumerate(users) if u.cell == k]
            est, edges = {}, set()
            for i in mine:
                u = users[i]
                ports = [(u.port0 + l - u.sc_start) % cell.comb for l in range(u.n_layers)]
                part = Y[:, u.sc_start:u.sc_start + u.sc_count]
                est[i] = _x_ls(part, pils[i], ports, cell.comb, False).mean(0)           # [L, n, B]
                edges |= {u.sc_start, u.sc_start + u.sc_count}
            edges = sorted(edges)
            for a0, a1 in zip(edges, edges[1:]):
                on = [i for i in mine if users[i].sc_start <= a0 and a1 <= users[i].sc_start + users[i].sc_count]
                if not on:
                    continue
                H = torch.cat([est[i][:, a0 - users[i].sc_start:a1 - users[i].sc_start] for i in on]).transpose(0, 1)
                x = _x_solve(H, Y[list(_DATA)][:, a0:a1], cell.noise_var)
                o = 0
                for i in on:
                    u = users[i]
                    xs[i][:, :, a0 - u.sc_start:a1 - u.sc_start] = x[o:o + u.n_layers]
                    o += u.n_layers
        return {"x_hat": torch.cat([x.reshape(-1) for x in xs]), "bits": None, "status": None}
    if kind == "cnn":
        beam, pil = _detect_inputs(c, seed)
        p = torch.load(_WEIGHTS, map_location="cpu")["params"].cuda().to(torch.bfloat16).double()
        L, Bm, n_sc, nv = c["n_layers"], c["n_beams"], c["n_sc"], 10.0 ** (-c["snr_db"] / 10.0)
        Hs, rs = [], []
        for i in range(c["n_slots"]):
            Y = beam[i].to(torch.complex128)
            E = _x_ls(Y, pil[i], range(L), L, False)                                    # [2, L, n_sc, B]
            v = E.permute(1, 3, 0, 2).reshape(L * Bm, 2, n_sc)
            sc = v.abs().square().mean(dim=(1, 2)).sqrt()[:, None, None, None]
            x = torch.stack([v.real, v.imag], dim=1) / sc                               # [grids, 2 ch, 2 rows, n_sc]
            y = torch.cat([_x_forward(x[k:k + 64], p)[0] for k in range(0, x.shape[0], 64)]) * sc
            y = torch.complex(y[:, 0], y[:, 1]).reshape(L, Bm, 2, n_sc)
            H = E.mean(0).clone()                                                       # [L, n_sc, B]
            for l in range(L):
                k = torch.arange(l, n_sc, L, device="cuda")
                z = (Y[list(_DMRS)][:, k] / pil[i][l][:, k].to(torch.complex128)[..., None]).permute(2, 0, 1)  # [B, 2, K]
                r_cnn = (z - y[l][:, :, k]).abs().square().mean(dim=(1, 2))
                r_loo = (z[:, :, 1:-1] - 0.5 * (z[:, :, :-2] + z[:, :, 2:])).abs().square().mean(dim=(1, 2))
                r = r_cnn / r_loo.clamp(min=nv)
                rs.append(r)
                use = r <= 2.0
                H[l][:, use] = y[l].mean(1).T[:, use]
            Hs.append(H.transpose(0, 1))
        return {"H": torch.stack(Hs), "resid": torch.cat(rs), "fallback": None}
    x, target, p0, m0, v0 = _train_inputs(c, seed)
    pb = p0.to(torch.bfloat16).double().requires_grad_(True)
    n, w = c["n_grids"], c["width"]
    ys, acts, loss = [], [], 0.0
    grad = torch.zeros_like(pb)
    for k in range(0, n, 64):
        y, a = _x_forward(x[k:k + 64].double(), pb)
        part = (y - target[k:k + 64].double()).square().sum() / (n * 4 * w)
        grad += torch.autograd.grad(part, pb)[0]
        loss += float(part.detach())
        ys.append(y.detach())
        acts.append(torch.stack([v.detach().float() for v in a]))
    m = 0.9 * m0.double() + 0.1 * grad
    v = 0.999 * v0.double() + 0.001 * grad.square()
    p = p0.double() - 1e-3 * (m / (1 - 0.9 ** 200)) / ((v / (1 - 0.999 ** 200)).sqrt() + 1e-8)
    return {"y": torch.cat(ys), "acts": torch.cat(acts, dim=1), "loss": torch.tensor([loss], dtype=torch.float64),
            "grad": grad, "p": p, "pb": p, "m": m, "v": v}
