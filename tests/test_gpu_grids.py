"""How many CTAs the convolution runs with, as the profiler of torch sees the launches."""
import json

import numpy as np
import pytest

from paper_1912_11040_b200 import binding, synth

pytestmark = pytest.mark.gpu


def convolve_grids(call, tmp_path):
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
    return [e["args"]["grid"][0] for e in launches if "convolve_kernel" in e["name"]]


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
        grids[staging] = convolve_grids(lambda: ctx.aug_pipeline(speech, w.stride, lengths, w.lengths, bank, w.bank.size,
                                                                 table, w.B, feats, T, counts), tmp_path)
    assert len(grids[False]) == 1 and grids[True] == grids[False]
