"""How many CTAs kernels run with, as the profiler of torch sees the launches."""
import json

import numpy as np
import pytest

from paper_1912_11040_b200 import binding, synth

pytestmark = pytest.mark.gpu


def grids_of(kernel, call, tmp_path):
    import torch
    call()
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    launches = [e for e in json.load(open(path))["traceEvents"] if "grid" in e.get("args", {})]
    if not launches:
        pytest.skip("the profiler sees no launches here")
    return [tuple(e["args"]["grid"]) for e in launches if kernel in e["name"]]


def test_device_calls_use_the_whole_device_in_every_context(tmp_path):
    """Room for the copying kernels of the host entry point is left by its chunks, not by device calls
    of a context that could be used for it."""
    import torch
    w = synth.make_workload(2, seed=1, batch=200, dur_scale=0.3)
    grids = {}
    for staging in (False, True):
        cfg = binding.make_config(w.cfg, w.B, w.stride, host_staging=staging, max_bank_samples=w.bank.size)
        ctx = binding.AugContext(cfg)
        cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        speech, lengths, bank, table = cu(w.speech), cu(w.lengths), cu(w.bank), binding.table_to_device(w.table)
        T = binding.aug_frame_count(int(w.lengths.max()), cfg.win, cfg.hop)
        feats = torch.empty((w.B, T, cfg.n_mel), device="cuda")
        counts = torch.empty(w.B, dtype=torch.int32, device="cuda")
        grids[staging] = grids_of("convolve_kernel", lambda: ctx.aug_pipeline(speech, w.stride, lengths, w.lengths, bank,
                                                                              w.bank.size, table, w.B, feats, T, counts),
                                  tmp_path)
    assert len(grids[False]) == 1 and grids[True] == grids[False]


def context(batch, samples, **fields):
    w = synth.make_workload(2, seed=1, batch=2, dur_scale=0.1)
    w.cfg.update(fields)
    return binding.AugContext(binding.make_config(w.cfg, batch, samples)), w.table


@pytest.mark.parametrize("win,hop,B,seconds,grid", [
    (400, 160, 3, 3, (10, 3, 1)),                    # single tiles of 32 frames: no arithmetic for a mixture
    (320, 320, 100, 10, (400, 1, 1)),                # 16 large tiles each: runs of four alone
    (400, 160, 100, 10, ((100 - 19) * 8 + 19 * 32, 1, 1))])      # 32 small ones: the last 19 utterances tile by tile
def test_tiles_of_the_power_spectra(win, hop, B, seconds, grid, tmp_path):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the numbers are those of 148 multiprocessors")
    n = seconds * 16000
    ctx, _ = context(B, n, n_fft=512, win=win, hop=hop)
    T = binding.aug_frame_count(n, win, hop)
    x, lengths = torch.zeros((B, n), device="cuda"), torch.full((B,), n, dtype=torch.int32, device="cuda")
    power, counts = torch.empty((B, T, 257), device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda")
    assert grids_of("frames_kernel", lambda: ctx.feat_stft_power(x, n, lengths, B, power, T, counts), tmp_path) == [grid]


def test_few_long_utterances_are_warped_in_runs(tmp_path):
    import torch
    B, n = 4, 1600000
    ctx, table = context(B, n, vtlp_win=400)
    x, lengths = torch.zeros((B, n), device="cuda"), torch.full((B,), n, dtype=torch.int32, device="cuda")
    out, rows = torch.empty_like(x), binding.table_to_device(np.tile(table[:1], B))
    got = grids_of("vtlp_resynth_kernel", lambda: ctx.aug_vtlp_resynth(x, n, lengths, rows, B, out, n), tmp_path)
    hops = (n + 300 + 99) // 100
    assert got == [(B * ((hops + 44) // 45), 1, 1)]
