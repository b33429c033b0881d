"""The separate feature stages at the edges of their tiles: cepstra, mean and variance,
filterbank on given power spectra -- against the fp64 checker."""
import numpy as np
import pytest

import oracle
from paper_1912_11040_b200 import binding, synth

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24


def context(B, n_mel, n_fft=512):
    cfg = binding.AugConfig(fs=16000, win=400, hop=160, n_fft=n_fft, n_mel=n_mel, f_lo=0.0, f_hi=8000.0,
                            rir_taps=64, max_order=1, max_sources=1, frac_half_width=40, sound_speed=343.0,
                            log_floor=1e-7, pad_value=-3.5, compression=binding.COMPRESS_LOG, max_batch=B,
                            max_samples=16000, host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0,
                            host_rows=0)
    return binding.AugContext(cfg)


def draw(B, T_max, D, seed):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((B, T_max, D)) * 2.0 - 5.0).astype(np.float32)
    counts = rng.integers(0, T_max + 1, B).astype(np.int32)
    counts[0] = T_max
    if B > 1:
        counts[1] = 0
    return x, counts


# tile edges (128 frames), odd band counts, more than one round of 16 coefficients, one band
@pytest.mark.parametrize("T_max,M,n_cep", [(1, 40, 13), (127, 80, 13), (128, 23, 23), (129, 128, 128),
                                           (300, 64, 17), (65, 1, 1), (257, 40, 16)])
def test_mfcc_tiles(T_max, M, n_cep):
    import torch
    B = 3
    x, counts = draw(B, T_max, M, T_max + M)
    out = torch.full((B, T_max, n_cep), float("nan"), device="cuda")
    ctx = context(B, M)
    ctx.feat_mfcc(torch.from_numpy(x).cuda(), torch.from_numpy(counts).cuda(), B, T_max, n_cep, out)
    got = out.cpu().numpy()
    for b in range(B):
        T = counts[b]
        assert np.all(got[b, T:] == -3.5)
        if T:
            # M products and sums of fp32 numbers; a basis value is off by pi (its angle, reduced exactly, is rounded
            # once below 2 half turns), the cosine's own error, the scale's and the product's: 8 units
            bound = (M + 8) * EPS * np.sqrt(2.0 / M) * np.abs(x[b, :T]).sum(1, keepdims=True)
            assert np.all(np.abs(got[b, :T] - oracle.mfcc(x[b, :T], n_cep)) <= bound)


# one column, columns that do not fill the CTA, rows of 16-byte multiples, more columns than a round
@pytest.mark.parametrize("T_max,D", [(1, 1), (5, 3), (33, 80), (700, 23), (97, 256), (40, 300), (9, 1028),
                                     (3001, 4)])
def test_mean_var_shapes(T_max, D):
    import torch
    B = 3
    x, counts = draw(B, T_max, D, T_max + D)
    mean = torch.full((B, D), float("nan"), device="cuda")
    var = torch.full_like(mean, float("nan"))
    context(B, 40).feat_mean_var(torch.from_numpy(x).cuda(), torch.from_numpy(counts).cuda(), B, T_max, D, mean, var)
    mean, var = mean.cpu().numpy(), var.cpu().numpy()
    for b in range(B):
        T = counts[b]
        if T == 0:
            assert not mean[b].any() and not var[b].any()
            continue
        y = x[b, :T].astype(np.float64)
        mu = y.mean(0)
        # fp64 sums, one rounding to fp32; the variance is a difference of fp64 sums of about mu^2 + var
        assert np.all(np.abs(mean[b] - mu) <= 2 * EPS * np.abs(mu))
        vr = y.var(0)
        assert np.all(np.abs(var[b] - vr) <= 2 * EPS * vr + 4 * T * 2.0 ** -53 * (mu * mu + vr))


# rows that start at any offset from a 16-byte boundary, tiles of 32 frames, widest and narrowest bands
@pytest.mark.parametrize("T_max,M,n_fft", [(1, 40, 512), (31, 80, 512), (33, 128, 1024), (66, 1, 512), (35, 23, 1024)])
def test_logmel_tiles(T_max, M, n_fft):
    import torch
    B = 3
    rng = np.random.default_rng(T_max + M)
    K = n_fft // 2 + 1
    P = np.exp(rng.standard_normal((B, T_max, K)) * 3.0).astype(np.float32)
    counts = np.array([T_max, 0, T_max // 2], dtype=np.int32)
    tab = np.zeros(B, dtype=synth.UTT_DTYPE)
    tab["alpha"] = [1.0, 0.9, 1.13]
    out = torch.full((B, T_max, M), float("nan"), device="cuda")
    ctx = context(B, M, n_fft)
    ctx.feat_vtlp_logmel(torch.from_numpy(P).cuda(), torch.from_numpy(counts).cuda(), binding.table_to_device(tab),
                         B, T_max, out)
    got = out.cpu().numpy()
    for b in range(B):
        T = counts[b]
        assert np.all(got[b, T:] == -3.5)
        if T:
            ref = oracle.logmel(P[b, :T].astype(np.float64), float(tab["alpha"][b]), n_fft, M, floor=1e-7)
            # positive terms: relative error of a sum of K of them, plus that of the logarithm
            assert np.all(np.abs(got[b, :T] - ref) <= (K + 4) * EPS + 4 * EPS * np.abs(ref))


# the waveform written by the feature kernel: full and single tiles, hops that are no multiple of 4,
# both transforms, and the pass of its own where frames leave gaps; utterances without a frame
@pytest.mark.parametrize("n_fft,win,hop,batch", [(512, 400, 160, 7), (512, 400, 160, 300), (512, 401, 125, 7),
                                                 (512, 160, 160, 7), (512, 200, 300, 7), (1024, 800, 200, 300)])
def test_waveform_written_with_the_features(n_fft, win, hop, batch):
    import torch
    w = synth.make_workload(2, seed=1, batch=7, dur_scale=0.12)
    w.lengths[1], w.lengths[2], w.lengths[3] = 0, win - 1, win
    rep = lambda a: np.ascontiguousarray(np.tile(a, (-(-batch // 7),) + (1,) * (a.ndim - 1))[:batch])
    speech, lengths, table = rep(w.speech), rep(w.lengths), rep(w.table)
    w.cfg.update(n_fft=n_fft, win=win, hop=hop)
    cfg = binding.make_config(w.cfg, batch, w.stride)
    ctx = binding.AugContext(cfg)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d_speech, d_len, d_bank, d_tab = cu(speech), cu(lengths), cu(w.bank), binding.table_to_device(table)
    T = binding.aug_frame_count(int(lengths.max()), win, hop)
    feats = torch.empty((batch, T, cfg.n_mel), device="cuda")
    wave = torch.full((batch, w.stride), float("nan"), device="cuda")
    ctx.aug_pipeline(d_speech, w.stride, d_len, lengths, d_bank, w.bank.size, d_tab, batch, feats, T,
                     torch.empty(batch, dtype=torch.int32, device="cuda"), wave)
    # the separate steps: responses, convolution and mix
    rir = torch.empty((batch, cfg.max_sources, cfg.rir_taps), device="cuda")
    ctx.aug_rir_image_method(d_tab, batch, rir)
    ref = torch.full_like(wave, float("nan"))
    ctx.aug_reverb_mix(d_speech, w.stride, d_len, d_bank, w.bank.size, rir, d_tab, batch, ref)
    wave, ref = wave.cpu().numpy(), ref.cpu().numpy()
    for b in range(batch):
        n = int(lengths[b])
        # same arithmetic but for the order in which the blocks' energies are added (fp64, then one
        # fp32 rounding of the gain): two roundings of the sum of both sides
        if n:
            assert np.max(np.abs(wave[b, :n] - ref[b, :n])) <= 4 * EPS * np.max(np.abs(ref[b, :n]))
        assert np.all(np.isnan(wave[b, n:]))


@pytest.mark.parametrize("rows", [1, 40, 0])
def test_waveform_with_fewer_feature_rows_than_frames(rows):
    """The waveform does not depend on how many feature rows are asked for; where most of it lies
    behind the last row, it has a launch of its own instead of one CTA's loop.  rows = 0: all."""
    import torch
    from helpers import Device
    dev = Device(synth.make_workload(2, seed=3, batch=5, dur_scale=0.2))
    _, _, ref = dev.pipeline()
    before = dev.ctx.aug_launch_count()
    _, _, full = dev.pipeline()
    base = dev.ctx.aug_launch_count() - before
    F, counts, wave = dev.pipeline(T_max=rows or dev.T_max, lengths_host=False)
    launches = dev.ctx.aug_launch_count() - before - base
    assert launches == base + (1 if rows else 0)
    assert int(counts.max()) == (rows or dev.T_max)
    wave, ref = wave.cpu().numpy(), ref.cpu().numpy()
    for b in range(dev.w.B):
        n = int(dev.w.lengths[b])
        # the gain's energies are added in another order: two roundings of the sum of both sides
        assert np.max(np.abs(wave[b, :n] - ref[b, :n])) <= 4 * EPS * np.max(np.abs(ref[b, :n]))
        assert np.all(np.isnan(wave[b, n:]))


@pytest.mark.parametrize("n_fft,hop", [(512, 160), (512, 125), (1024, 200)])
def test_noise_that_is_not_finite_shows_in_the_waveform_alone(n_fft, hop):
    """Infinite or undefined noise makes the gain 0; the waveform is still y_s + 0 v, undefined where v is
    and in all of the utterance alike, as the separate mix gives it, and the features are those of y_s."""
    import torch
    from helpers import LOGMEL_ABS_TOL, Device
    w = synth.make_workload(2, seed=5, batch=3, dur_scale=0.2)
    w.cfg.update(n_fft=n_fft, win=400, hop=hop)
    w.table["n_src"][:] = [2, 1, 2]
    clean = synth.Workload(name=w.name, cfg=w.cfg, lengths=w.lengths, speech=w.speech, bank=w.bank, table=w.table.copy())
    clean.table["n_src"][:] = 1
    F_ref, _, _ = Device(clean).pipeline()
    for bad in (np.nan, np.inf):
        o, m = int(w.table["noise_offset"][0, 0]), int(w.table["noise_len"][0, 0])
        w.bank = w.bank.copy()
        w.bank[o:o + m] = bad
        dev = Device(w)
        F, _, wave = dev.pipeline()
        mixed = dev.reverb_mix(dev.rir())
        assert torch.equal(torch.isnan(wave), torch.isnan(mixed))
        assert torch.isnan(wave[0, : int(w.lengths[0])]).all() and torch.isfinite(wave[1, : int(w.lengths[1])]).all()
        # the same y_s from blocks of other sizes (they follow the longest response of an utterance): each side
        # is within LOGMEL_ABS_TOL of the exact features
        assert (F[0] - F_ref[0]).abs().max() <= 2 * LOGMEL_ABS_TOL


@pytest.mark.parametrize("n_fft,hop", [(512, 160), (512, 125), (1024, 200)])
def test_noise_whose_energy_overflows_shows_in_the_waveform_alone(n_fft, hop):
    """Noise so loud that the sum of its squares is infinite makes the gain 0, and the features are those of y_s, also
    where single samples of v overflow and the others do not: a click at levels up to the largest float."""
    import torch
    from helpers import LOGMEL_ABS_TOL, Device
    w = synth.make_workload(2, seed=5, batch=2, dur_scale=0.2)
    w.cfg.update(n_fft=n_fft, win=400, hop=hop)
    w.table["n_src"][:] = [2, 1]
    w.table["noise_weight"][0, 0] = 50.0
    clean = synth.Workload(name=w.name, cfg=w.cfg, lengths=w.lengths, speech=w.speech, bank=w.bank, table=w.table.copy())
    clean.table["n_src"][:] = 1
    F_ref, _, _ = Device(clean).pipeline()
    o, m = int(w.table["noise_offset"][0, 0]), int(w.table["noise_len"][0, 0])
    lone = 0
    for level in 1e36 * 1.2 ** np.arange(30):
        w.bank = np.zeros_like(w.bank)
        w.bank[o + m // 2] = level
        F, _, wave = Device(w).pipeline()
        wrong = int((~torch.isfinite(wave[0, : int(w.lengths[0])])).sum())
        lone += 0 < wrong < 1000
        # each side is within LOGMEL_ABS_TOL of the exact features
        assert (F[0] - F_ref[0]).abs().max() <= 2 * LOGMEL_ABS_TOL, (level, wrong)
    assert lone > 0


# tiles that begin at any sample of a 16-byte group: rows of whole groups are copied in one tile ahead, other
# rows sample by sample; single tiles and runs of them, last tiles of any number of frames
@pytest.mark.parametrize("n_fft,win,hop", [(512, 400, 125), (512, 401, 110), (512, 3, 1), (512, 77, 131),
                                           (1024, 500, 441), (1024, 1023, 163), (512, 400, 900), (512, 511, 513),
                                           (1024, 1024, 1022), (1024, 801, 1599)])
@pytest.mark.parametrize("batch", [3, 200])
def test_power_spectra_of_rows_that_start_anywhere(n_fft, win, hop, batch):
    import torch
    T_max = 170
    n = (T_max - 1) * hop + win + 5
    rng = np.random.default_rng(win + hop)
    lengths = rng.integers(0, n + 1, batch).astype(np.int32)
    lengths[:3] = n, n - hop - 6, min(win + 31 * hop, n)
    wave = rng.standard_normal((batch, n)).astype(np.float32)
    for b in range(batch):
        wave[b, lengths[b]:] = np.nan                  # nothing beyond an utterance's end is used
    cfg = binding.AugConfig(fs=16000, win=win, hop=hop, n_fft=n_fft, n_mel=40, f_lo=0.0, f_hi=8000.0, rir_taps=64,
                            max_order=1, max_sources=1, frac_half_width=40, sound_speed=343.0, log_floor=1e-7,
                            pad_value=-3.5, compression=binding.COMPRESS_LOG, max_batch=batch, max_samples=n + 8,
                            host_staging=0, image_lattice=0, max_bank_samples=0, vtlp_win=0, host_rows=0)
    ctx = binding.AugContext(cfg)
    got = []
    for stride in ((n + 3) // 4 * 4, (n + 3) // 4 * 4 + 1):
        x = torch.full((batch, stride), float("nan"), device="cuda")
        x[:, :n] = torch.from_numpy(wave)
        P = torch.full((batch, T_max, n_fft // 2 + 1), float("nan"), device="cuda")
        counts = torch.full((batch,), -7, dtype=torch.int32, device="cuda")
        ctx.feat_stft_power(x, stride, torch.from_numpy(lengths).cuda(), batch, P, T_max, counts)
        got.append((P.cpu().numpy(), counts.cpu().numpy()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    P, counts = got[0]
    for b in range(3):
        T = min(binding.aug_frame_count(int(lengths[b]), win, hop), T_max)
        assert counts[b] == T and not P[b, T:].any()
        ref = oracle.stft_power(wave[b, : lengths[b]].astype(np.float64), win, hop, n_fft)[:T]
        if T:
            # two frames share a transform of 9 (10) levels: a few roundings of the loudest bin around
            assert np.max(np.abs(P[b, :T] - ref)) <= 2e-6 * ref.max()


@pytest.mark.parametrize("n_fft,win,hop", [(512, 200, 600), (512, 512, 1022), (1024, 1024, 1000), (1024, 1024, 1024),
                                           (1024, 801, 1603), (1024, 400, 3001), (1024, 400, 6188)])
def test_hops_beyond_the_window(n_fft, win, hop):
    """Tiles whose samples, with the gaps between frames, fit no buffer for copying ahead, up to the
    largest hop that is served; one more is refused."""
    from helpers import Device, check_pipeline_against_oracle, oracle_batch
    w = synth.make_workload(1, seed=hop, batch=3, dur_scale=9.0 if hop > 2000 else 4.0)
    w.cfg.update(n_fft=n_fft, win=win, hop=hop)
    w.lengths[1], w.lengths[2] = win + 4 * hop + 1, win
    dev = Device(w)
    F, counts, wave = dev.pipeline()
    check_pipeline_against_oracle(dev, F, counts, wave, oracle_batch(w))
    if hop == 6188:
        w.cfg.update(hop=hop + 1)
        with pytest.raises(binding.AugError) as e:
            Device(w).pipeline()
        assert e.value.code == binding.AUG_ECAP
        with pytest.raises(binding.AugError):
            Device(w).stft_power(dev.speech)


@pytest.mark.parametrize("n_fft", [512, 1024])
def test_power_spectra_do_not_depend_on_the_place_in_the_batch(n_fft):
    """A batch of which the first utterances are done in runs of tiles and the last ones tile by tile: copies of an utterance
    come out bit by bit the same wherever they stand, with lengths around a tile, a run, and none."""
    import torch
    lengths = np.array([20000, 400 + 31 * 160, 400 + 32 * 160, 399, 0, 400 + 127 * 160 + 3], np.int32)
    few, B, stride = len(lengths), 420, 20732
    rng = np.random.default_rng(n_fft)
    wave = (rng.standard_normal((few, stride)) * 0.05).astype(np.float32)
    w = synth.make_workload(1, batch=2, dur_scale=0.1)
    w.cfg.update(n_fft=n_fft)
    ctx = binding.AugContext(binding.make_config(w.cfg, B, stride))
    T = binding.aug_frame_count(int(lengths.max()), 400, 160)
    rep = lambda a: torch.from_numpy(np.tile(a, (B // few,) + (1,) * (a.ndim - 1))).cuda()
    power = torch.full((B, T, n_fft // 2 + 1), float("nan"), device="cuda")
    counts = torch.full((B,), -1, dtype=torch.int32, device="cuda")
    ctx.feat_stft_power(rep(wave), stride, rep(lengths), B, power, T, counts)
    first = power[:few].repeat(B // few, 1, 1)
    assert torch.equal(power, first)
    assert counts.cpu().tolist() == [binding.aug_frame_count(int(n), 400, 160) for n in lengths] * (B // few)
    ref = oracle.stft_power(wave[0, :20000].astype(np.float64), 400, 160, n_fft)
    got = power[0, : len(ref)].cpu().numpy()
    # amplitudes within a few roundings of the largest one, squared
    assert np.max(np.abs(got - ref)) <= 32 * EPS * np.max(ref)
