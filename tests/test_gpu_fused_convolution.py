"""The convolution where its blocks, loads and work list have edges, against the fp64
checker: utterances that end with a block, one sample around it, within the first group of
four; noise stretches at every offset from a 16-byte boundary, read inside one period, across
its end, and looped many times; more units of work than resident CTAs, on every route."""
import numpy as np
import pytest

import oracle
from paper_1912_11040_b200 import binding, synth
from helpers import check_wave

pytestmark = pytest.mark.gpu
TAPS = 300
OB = (16384 - TAPS + 1) & ~3         # outputs per block


def run(lengths, stretches, taps=TAPS, seed=0, copies=1, calls=1, hold=False):
    """stretches[b] = list of (offset, length); responses dense over `taps`; SNRs of -4 to 8 dB, so that every
    utterance's noise is at least 0.4 of its waveform, thousands of times what check_wave allows.  The batch holds every
    utterance `copies` times and goes through the same context `calls` times; every result is compared."""
    import torch
    rng = np.random.default_rng(seed)
    B, S = len(lengths), 1 + max(len(s) for s in stretches)
    stride = (max(lengths) + 3) // 4 * 4
    bank = (rng.standard_normal(max([60000] + [o + m for s in stretches for o, m in s])) * 0.05).astype(np.float32)
    speech = np.zeros((B, stride), np.float32)
    tab = np.zeros(B, dtype=synth.UTT_DTYPE)
    rir = np.zeros((B, S, taps), np.float32)
    for b, n in enumerate(lengths):
        speech[b, :n] = rng.standard_normal(n) * 0.05
        tab[b]["n_src"], tab[b]["snr_db"] = 1 + len(stretches[b]), 3.0 * (b % 5) - 4.0
        for k, (o, m) in enumerate(stretches[b]):
            tab[b]["noise_offset"][k], tab[b]["noise_len"][k], tab[b]["noise_weight"][k] = o, m, 1.0 - 0.3 * k
        rir[b, : tab[b]["n_src"]] = rng.standard_normal((tab[b]["n_src"], taps)) * np.exp(-np.arange(taps) / (0.3 * taps)) * 0.1
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=512, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=taps,
                            max_order=1, max_sources=S, frac_half_width=40, sound_speed=343.0, log_floor=1e-7,
                            pad_value=0.0, compression=binding.COMPRESS_LOG, max_batch=B * copies,
                            max_samples=stride, host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0,
                            host_rows=0)
    ctx = binding.AugContext(cfg)
    if hold:
        ctx.aug_hold_parking_slots(True)
    rep = lambda a: np.tile(a, (copies,) + (1,) * (a.ndim - 1))
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    args = [cu(rep(speech)), stride, cu(rep(np.array(lengths, np.int32))), cu(bank), bank.size, cu(rep(rir)),
            binding.table_to_device(rep(tab)), B * copies]
    got = []
    for _ in range(calls):
        out = torch.full((B * copies, stride), float("nan"), device="cuda")
        ctx.aug_reverb_mix(*args, out)
        torch.cuda.synchronize()
        got += list(out.cpu().numpy().reshape(copies, B, stride))
    for b, n in enumerate(lengths):
        noises = [oracle.looped_noise(bank, o, m, n) for o, m in stretches[b]]
        ref, *_ = oracle.reverb_mix(speech[b, :n].astype(np.float64),
                                    [rir[b, s].astype(np.float64) for s in range(int(tab[b]["n_src"]))], noises,
                                    tab[b]["noise_weight"], tab[b]["snr_db"])
        for i, g in enumerate(got):
            check_wave(g[b, :n], ref, f"utt {b} of {n} samples, copy {i}")
            assert np.all(np.isnan(g[b, n:]))


def test_lengths_around_a_block():
    lengths = [OB, OB - 1, OB + 1, 2 * OB + 3, 3, 1, 401]
    run(lengths, [[(8, 5000)]] * len(lengths))


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_stretches_at_any_offset(offset):
    """50003 samples: blocks that lie inside the stretch, across its end, and at both ends of
    the utterance; the short ones wrap inside a block; lengths that are multiples of 4 and not."""
    lengths = [50003, 50003, 40000, 33000]
    run(lengths, [[(100 + offset, 40000 + offset)], [(offset, 44000), (7 + offset, 321)], [], [(4 + offset, 7 + offset)]],
        seed=offset)


def test_more_units_than_resident_ctas():
    """600 utterances of one block, both outputs: most units are drawn from the counter."""
    rng = np.random.default_rng(4)
    lengths = [int(n) for n in rng.integers(1, 900, 600)]
    run(lengths, [[(4 * (b % 50), 200 + b)] if b % 3 else [] for b in range(600)], taps=50)


@pytest.mark.parametrize("taps", [8193, 16385, 24576])
def test_long_responses_with_many_units(taps):
    """The stored-spectra route: lengths around its blocks of 8192, several units a CTA in each of its
    kernels; the first call of a context launches the fused kernels too, the later ones know better."""
    lengths = [8192 * k + d for k in (1, 2, 4) for d in (-1, 0, 1)] + [49153]
    loops = [[(8, 40000)], [(5, 8193), (4, 16384)], []]
    run(lengths, [loops[b % 3] for b in range(len(lengths))], taps=taps, copies=16, calls=3)


@pytest.mark.parametrize("hold", [False, True])
def test_parking_slots_used_by_many_units(hold):
    """Three noise sources, several units a CTA: a slot is written again by the unit after."""
    run([3 * OB + 5, 2 * OB, 700], [[(8, 40000), (3, 9000), (100, 777)], [(0, 50000), (16, 20000)],
                                    [(4, 400), (1, 333), (7, 50)]], copies=80, calls=2, hold=hold)


@pytest.mark.parametrize("taps", [1, 300, 8192])
def test_noise_that_comes_back(taps):
    """One noise source whose stretch is shorter than the utterance: only the blocks up to the end of its first period
    (and of the response behind it) are computed.  Periods of any alignment, around the length of a block, of
    the utterance and far below, utterances that end right behind the computed blocks; a second noise, which needs all of them."""
    ob = (16384 - taps + 1) & ~3
    lengths, loops = [], []
    for n in (6 * ob, 6 * ob + 1, 5 * ob - 3, 60001):
        for m in (ob, ob + 1, ob - 2, 2 * ob - taps + 1, 2 * ob - taps + 2, 3 * ob + 3, 1, 3, 4, 1000, 1001, n - 1, n, n + 1):
            lengths.append(n)
            loops.append([(8 + len(loops) % 3, max(m, 1))])
    lengths.append(6 * ob + 1)
    loops.append([(8, 2 * ob), (4, ob)])
    run(lengths, loops, taps=taps, seed=taps)


def test_energy_of_noise_that_comes_back():
    """The gain of a stretch that is repeated up to a million times: the mix has the SNR that was asked for.  A constant
    stretch, so that errors of equal terms add up instead of averaging out."""
    import torch
    n, taps, snr = 960003, TAPS, -6.0
    stretches = [1, 3, 4, 1000, 1001, OB, 3 * OB + 1, n // 2 - 1, n // 2, n]
    B, stride = len(stretches), (n + 3) // 4 * 4
    rng = np.random.default_rng(7)
    bank = torch.full((n,), 0.05, device="cuda")
    speech = torch.from_numpy((rng.standard_normal((B, stride)) * 0.05).astype(np.float32)).cuda()
    rir = torch.from_numpy(np.abs(rng.standard_normal((B, 2, taps))).astype(np.float32) * 0.01).cuda()
    tab = np.zeros(B, dtype=synth.UTT_DTYPE)
    tab["snr_db"], tab["noise_len"][:, 0], tab["noise_weight"][:, 0] = snr, stretches, 1.0
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=512, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=taps,
                            max_order=1, max_sources=2, frac_half_width=40, sound_speed=343.0, log_floor=1e-7,
                            pad_value=0.0, compression=binding.COMPRESS_LOG, max_batch=B, max_samples=stride,
                            host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0, host_rows=0)
    ctx = binding.AugContext(cfg)
    lengths = torch.full((B,), n, dtype=torch.int32, device="cuda")
    out = []
    for n_src in (1, 2):
        tab["n_src"] = n_src
        w = torch.full((B, stride), float("nan"), device="cuda")
        ctx.aug_reverb_mix(speech, stride, lengths, bank, n, rir, binding.table_to_device(tab), B, w)
        out.append(w[:, :n].double())
    y, noise = out[0], out[1] - out[0]
    got = y.square().sum(1) / noise.square().sum(1) / 10.0 ** (snr / 10.0)
    # each of the two sums: 16 roundings a lane of the packed sum, as many of the copies', seven to add up a warp's; the
    # gain's and the wave's
    bound = (2 * 39 + 2 + 2) * 2.0 ** -24
    assert (got - 1.0).abs().max() <= bound, (got - 1.0).tolist()


@pytest.mark.parametrize("copies", [1, 8])
def test_short_stretches_take_no_longer_than_long_ones(copies):
    """One and eight utterances of 60 s: noise that comes back sixty times is no more work than noise that does not."""
    import torch
    n, taps = 960000, 4001
    stride = n
    rng = np.random.default_rng(3)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    bank, speech = cu(rng.standard_normal(n) * 0.05), cu(rng.standard_normal((copies, stride)) * 0.05)
    rir = cu(rng.standard_normal((copies, 2, taps)) * 0.01)
    lengths = torch.full((copies,), n, dtype=torch.int32, device="cuda")
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=512, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=taps,
                            max_order=1, max_sources=2, frac_half_width=40, sound_speed=343.0, log_floor=1e-7,
                            pad_value=0.0, compression=binding.COMPRESS_LOG, max_batch=copies, max_samples=stride,
                            host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0, host_rows=0)
    ctx, out = binding.AugContext(cfg), torch.empty((copies, stride), device="cuda")
    took = {}
    for m in (n, 16000, 16001):
        tab = np.zeros(copies, dtype=synth.UTT_DTYPE)
        tab["n_src"], tab["noise_len"][:, 0], tab["noise_weight"][:, 0] = 2, m, 1.0
        table, times = binding.table_to_device(tab), []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(8):
                ctx.aug_reverb_mix(speech, stride, lengths, bank, n, rir, table, copies, out)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        took[m] = min(times)
    # (a quarter for what a loaded machine adds; it was twice to ten times as long)
    assert max(took[16000], took[16001]) <= 1.25 * took[n], took
