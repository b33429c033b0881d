"""The waveform warp in runs of several rounds per CTA: batches large enough for them, windows
whose hop is a multiple of four (samples are added four at a time), even, and odd, the longest
window, utterances that end inside every part of a run."""
import numpy as np
import pytest

import oracle
from paper_1912_11040_b200 import binding, synth
from helpers import check_wave

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("win,n_max,B", [(64, 9000, 64), (60, 9000, 64), (56, 3001, 200), (800, 30000, 160),
                                         (1024, 13000, 600)])
def test_runs_of_rounds(win, n_max, B):
    import torch
    rng = np.random.default_rng(win)
    lengths = rng.integers(1, n_max + 1, B).astype(np.int32)
    lengths[0], lengths[1] = n_max, 0
    stride = (n_max + 3) // 4 * 4
    speech = (rng.standard_normal((B, stride)) * 0.05).astype(np.float32)
    tab = np.zeros(B, dtype=synth.UTT_DTYPE)
    tab["alpha"] = rng.uniform(0.8, 1.2, B)
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=512, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=64,
                            max_order=1, max_sources=1, frac_half_width=40, sound_speed=343.0, log_floor=1e-7,
                            pad_value=0.0, compression=binding.COMPRESS_LOG, max_batch=B, max_samples=stride,
                            host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=win, host_rows=0)
    ctx = binding.AugContext(cfg)
    out = torch.full((B, stride), float("nan"), device="cuda")
    ctx.aug_vtlp_resynth(torch.from_numpy(speech).cuda(), stride, torch.from_numpy(lengths).cuda(),
                         binding.table_to_device(tab), B, out, stride)
    got = out.cpu().numpy()
    for b in [0, 1] + list(range(2, B, max(1, B // 12))):
        n = int(lengths[b])
        check_wave(got[b, :n], oracle.vtlp_resynth(speech[b, :n].astype(np.float64), float(tab[b]["alpha"]), win),
                   f"utt {b} of {n} samples")
        assert np.all(np.isnan(got[b, n:]))


def test_wave_of_a_warped_batch_keeps_the_callers_row_stride():
    """The mixed waveform of a call with the waveform warp goes to rows of the caller's stride, also in
    a context made for longer utterances."""
    import torch
    w = synth.make_workload(2, seed=0, batch=4, dur_scale=0.1)
    w.cfg["vtlp_win"] = 400
    waves = []
    for room in (0, 5000):
        cfg = binding.make_config(w.cfg, w.B, w.stride + room)
        ctx = binding.AugContext(cfg)
        cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        T = binding.aug_frame_count(int(w.lengths.max()), cfg.win, cfg.hop)
        feats = torch.empty((w.B, T, cfg.n_mel), device="cuda")
        wave = torch.full((w.B, w.stride), float("nan"), device="cuda")
        ctx.aug_pipeline(cu(w.speech), w.stride, cu(w.lengths), w.lengths, cu(w.bank), w.bank.size,
                         binding.table_to_device(w.table), w.B, feats, T,
                         torch.empty(w.B, dtype=torch.int32, device="cuda"), wave)
        waves.append(wave.cpu().numpy())
    for b in range(w.B):
        n = int(w.lengths[b])
        assert np.all(np.isfinite(waves[0][b, :n])) and np.all(np.isnan(waves[1][b, n:]))
        # same arithmetic; the gain's sums may be added in another order
        np.testing.assert_allclose(waves[1][b, :n], waves[0][b, :n], rtol=0, atol=1e-6 * np.abs(waves[0][b, :n]).max())


def test_accuracy_of_the_transforms():
    """Root mean square error of the warped waveform.  Each of the two transforms contributes 1.1e-7 of the
    signal (nine additions and a few products deep, every factor rounded once), windows, splits, interpolation
    and overlap the rest: 1.9e-7 in all.  Factors that are not rounded once show: 3.1e-7 with powers of one."""
    import torch
    w = synth.make_workload(2, seed=11, batch=6, dur_scale=0.4)
    w.cfg["vtlp_win"] = 800
    ctx = binding.AugContext(binding.make_config(w.cfg, w.B, w.stride))
    out = torch.zeros((w.B, w.stride), device="cuda")
    ctx.aug_vtlp_resynth(torch.from_numpy(w.speech).cuda(), w.stride, torch.from_numpy(w.lengths).cuda(),
                         binding.table_to_device(w.table), w.B, out, w.stride)
    got = out.cpu().numpy().astype(np.float64)
    err = ref2 = 0.0
    for b in range(w.B):
        n = int(w.lengths[b])
        ref = oracle.vtlp_resynth(w.speech[b, :n].astype(np.float64), float(w.table["alpha"][b]), 800)
        err += np.sum((got[b, :n] - ref) ** 2)
        ref2 += np.sum(ref ** 2)
    assert np.sqrt(err / ref2) <= 2.3e-7
