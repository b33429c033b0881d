"""The response kernel at the edges of its windows, buffers and CTA sizes: half widths on both
sides of 40 (where the window stops fitting two and a half taps a lane) and the smallest,
buffers shorter than a window, images that begin before or end behind the buffer, odd
numbers of images, and batches large enough for the 256-thread CTAs."""
import numpy as np
import pytest

import oracle
from paper_1912_11040_b200 import binding, synth
from helpers import RIR_REL_TOL, WAVE_REL_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half_w", [1, 16, 39, 40, 41, 47])
@pytest.mark.parametrize("taps,B", [(60, 3), (97, 3), (700, 3), (333, 600)])
def test_windows_and_buffers(half_w, taps, B):
    import torch
    rng = np.random.default_rng(half_w * taps + B)
    tab = np.zeros(B, dtype=synth.UTT_DTYPE)
    tab["n_src"], tab["order"] = 1, rng.integers(0, 4, B)
    for b in range(B):
        tab[b]["room"] = rng.uniform(0.8, 6.0, 3)
        tab[b]["beta"] = rng.uniform(0.2, 1.0, 6)
        tab[b]["mic"] = tab[b]["room"] * rng.uniform(0.1, 0.45, 3)
        tab[b]["src_pos"][0] = tab[b]["room"] * rng.uniform(0.5, 0.9, 3)
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=512, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=taps,
                            max_order=3, max_sources=1, frac_half_width=half_w, sound_speed=343.0, log_floor=1e-7,
                            pad_value=0.0, compression=binding.COMPRESS_LOG, max_batch=B, max_samples=4,
                            host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0, host_rows=0)
    ctx = binding.AugContext(cfg)
    out = torch.full((B, 1, taps), float("nan"), device="cuda")
    ctx.aug_rir_image_method(binding.table_to_device(tab), B, out)
    h = out.cpu().numpy()[:, 0]
    for b in range(0, B, 1 if B < 10 else 29):
        r = tab[b]
        ref = oracle.rir_image_method(r["room"], r["beta"], r["mic"], r["src_pos"][0], int(r["order"]), taps,
                                      half_width=half_w)
        # fixed-point steps follow the direct path, which may lie behind a short buffer
        d0 = np.linalg.norm(r["mic"].astype(np.float64) - r["src_pos"][0])
        assert np.max(np.abs(h[b] - ref)) <= RIR_REL_TOL * max(np.max(np.abs(ref)), 1.0 / d0), b


@pytest.mark.parametrize("B,S,order", [(296, 1, 4), (297, 1, 4), (100, 3, 4), (90, 3, 5), (297, 1, 6), (297, 1, 10)])
def test_batches_on_both_sides_of_a_round(B, S, order):
    """Around the sizes from which smaller CTAs are taken (two 512-thread CTAs a multiprocessor): the responses
    do not depend on how many others are made."""
    import torch
    rng = np.random.default_rng(B + S + order)
    few, taps = 5, 1600
    tab = np.zeros(few, dtype=synth.UTT_DTYPE)
    tab["order"] = order
    tab["n_src"] = rng.integers(1, S + 1, few)
    for b in range(few):
        tab[b]["room"] = rng.uniform(3.0, 6.0, 3)
        tab[b]["beta"] = rng.uniform(0.5, 0.95, 6)
        tab[b]["mic"] = tab[b]["room"] * rng.uniform(0.1, 0.45, 3)
        for k in range(S):
            tab[b]["src_pos"][k] = tab[b]["room"] * rng.uniform(0.5, 0.9, 3)
    rows = np.tile(tab, -(-B // few))[:B]
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=512, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=taps,
                            max_order=order, max_sources=S, frac_half_width=40, sound_speed=343.0, log_floor=1e-7,
                            pad_value=0.0, compression=binding.COMPRESS_LOG, max_batch=B, max_samples=4,
                            host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0, host_rows=0)
    ctx = binding.AugContext(cfg)
    out = torch.full((B, S, taps), float("nan"), device="cuda")
    ctx.aug_rir_image_method(binding.table_to_device(rows), B, out)
    h = out.cpu().numpy()
    for b in range(few):
        for s in range(S):
            ref = np.zeros(taps)
            if s < tab[b]["n_src"]:
                r = tab[b]
                ref = oracle.rir_image_method(r["room"], r["beta"], r["mic"], r["src_pos"][s], order, taps)
            for i in range(b, B, few):
                assert np.max(np.abs(h[i, s] - ref)) <= RIR_REL_TOL * np.max(np.abs(ref)), (i, s)


@pytest.mark.parametrize("taps", [1000, 9000, 17000])
def test_ends_recorded_by_the_pipeline(taps):
    """What a context keeps from an earlier batch does not show: responses that end elsewhere, a source less, and a
    row that is rejected (silence) after a batch whose responses fill the buffer."""
    import torch
    w = synth.make_workload(2, seed=5, batch=6, dur_scale=0.15)
    w.cfg.update(rir_taps=taps)
    cfg = binding.make_config(w.cfg, w.B, w.stride)
    T = binding.aug_frame_count(int(w.lengths.max()), cfg.win, cfg.hop)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    speech, lengths, bank = cu(w.speech), cu(w.lengths), cu(w.bank)
    first, second = w.table.copy(), w.table.copy()
    first["beta"], first["room"] = 0.99, first["room"] * 1.5
    second["n_src"][1] = 1
    second["order"][2] = cfg.max_order + 1
    second["order"][3] = 0

    def run(ctx, table):
        feats = torch.full((w.B, T, cfg.n_mel), float("nan"), device="cuda")
        wave = torch.full((w.B, w.stride), float("nan"), device="cuda")
        ctx.aug_pipeline(speech, w.stride, lengths, w.lengths, bank, w.bank.size, binding.table_to_device(table), w.B,
                         feats, T, torch.empty(w.B, dtype=torch.int32, device="cuda"), wave)
        return wave.cpu().numpy()

    used, fresh = binding.AugContext(cfg), binding.AugContext(cfg)
    run(used, first)
    got, want = run(used, second), run(fresh, second)
    for b in range(w.B):
        n = int(w.lengths[b])
        # (after a batch of long responses the convolution goes another way: each within WAVE_REL_TOL of the definition)
        assert np.max(np.abs(got[b, :n] - want[b, :n])) <= 2 * WAVE_REL_TOL * np.sqrt(np.mean(want[b, :n] ** 2.0))
        assert (np.max(np.abs(got[b, :n])) == 0.0) == (b == 2)
