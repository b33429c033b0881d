"""The host entry point cuts a batch into chunks by the bytes it copies: few long utterances are
overlapped with their copies, many short ones are not torn into launches."""
import numpy as np
import pytest

from paper_1912_11040_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("utts,seconds,n_fft,n_mel,chunks", [
    (16, 60, 1024, 128, 8),       # 110 MB, the copies far longer than any launch
    (3, 60, 1024, 128, 2),        # 21 MB
    (1, 300, 512, 40, 1),         # 24 MB that cannot be cut
    (15, 19.99375, 512, 23, 2),   # 22 MB, chunks that begin at any feature row (an odd number of values)
    (24, 2, 512, 40, 1),          # 4 MB in many utterances
    (128, 2, 512, 40, 2)])        # 20 MB
def test_chunks_follow_the_bytes(utts, seconds, n_fft, n_mel, chunks):
    import torch
    w = synth.make_workload(1, seed=utts, batch=2, dur_scale=0.1)
    n = int(seconds * 16000)
    gen = torch.Generator().manual_seed(utts)
    speech = (torch.randn((utts, n), generator=gen) * 0.05).pin_memory()
    lengths = np.full(utts, n, np.int32)
    table = np.tile(w.table, -(-utts // 2))[:utts].copy()
    w.cfg.update(n_fft=n_fft, n_mel=n_mel)
    cfg = binding.make_config(w.cfg, utts, n, host_staging=True, max_bank_samples=w.bank.size)
    ctx = binding.AugContext(cfg)
    T = binding.aug_frame_count(n, cfg.win, cfg.hop)
    feats = torch.full((utts, T, n_mel), float("nan"), device="cuda")
    counts = torch.zeros(utts, dtype=torch.int32, device="cuda")
    cu = lambda a: torch.from_numpy(a).cuda()
    before = ctx.aug_launch_count()
    ctx.aug_pipeline(speech.cuda(), n, cu(lengths), lengths, cu(w.bank), w.bank.size, binding.table_to_device(table),
                     utts, feats, T, counts)
    torch.cuda.synchronize()
    one = ctx.aug_launch_count() - before
    out = torch.full((utts, T, n_mel), float("nan")).pin_memory()
    host_counts = torch.zeros(utts, dtype=torch.int32).pin_memory()
    ctx.aug_pipeline_host(speech, n, lengths, torch.from_numpy(w.bank), w.bank.size, table, utts, out, T, host_counts)
    # (rows of full length are copied by the copy engine alone: every launch is one of the pipeline's)
    assert ctx.aug_launch_count() - before - one == chunks * one
    assert torch.equal(host_counts, counts.cpu())
    # the same kernels; the gain's energies may be added in another order
    assert (out - feats.cpu()).abs().max() <= 1e-4
