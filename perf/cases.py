"""The work a training or evaluation job has this library do, as cases to time.

A job that trains on augmented speech keeps a context, a bank of noise recordings and a
stream; per batch it draws a parameter table on the host (`aug_sample_params`), has speech
on the GPU (or in pinned host memory) and calls `aug_pipeline` (or `aug_pipeline_host`).
Jobs that use one stage alone call that stage: responses (`aug_rir_image_method`), recorded
responses applied to speech (`aug_reverb_mix`), features of clean speech for evaluation
(`feat_stft_power`, `feat_vtlp_logmel`, `feat_mfcc`, `feat_mean_var`).

Sizes are those of the library's five synthetic workloads (2 s to 60 s utterances, 1 to 4096
of them, responses of 4096 to 24000 taps, one to three noises, 40 / 80 / 128 bands, 512- and
1024-point transforms) and what lies between them.  Lengths are ragged and odd.
"""
import math

import numpy as np
import torch

from paper_1912_11040_b200 import binding

FS = 16000
WIN, HOP = 400, 160          # 25 ms every 10 ms
HALF_WIDTH = 40              # 81-tap fractional delays


# ----------------------------------------------------------------------------- the cases
# Rooms, reverberation times, orders, SNRs and warp factors of the five workloads.
_STYLES = {
    #             rooms (m)                       T60 (s)    SNR (dB)   warp
    "office": dict(lo=(5, 4, 3), hi=(5, 4, 3), t60=(0.4, 0.4), snr=(10, 10), alpha=(0.9, 0.9)),
    "rooms": dict(lo=(3, 3, 3), hi=(10, 10, 10), t60=(0.1, 0.9), snr=(0, 30), alpha=(0.8, 1.2)),
    "far": dict(lo=(3, 3, 2.5), hi=(20, 15, 5), t60=(0.3, 1.5), snr=(-5, 20), alpha=(0.8, 1.2)),
    "halls": dict(lo=(4, 4, 4), hi=(12, 12, 12), t60=(0.3, 1.2), snr=(0, 20), alpha=(0.8, 1.2)),
}

_BASE = dict(call="pipeline", style="rooms", utts=1, min_s=2.0, max_s=2.0, taps=4096, order=6,
             noise_lo=1, noise_hi=1, noise_align=4, n_fft=512, n_mel=40, power_law=False,
             wave=False, vtlp_win=0)


def _case(name=None, **kw):
    c = dict(_BASE)
    c.update(kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one utterance as it arrives: an interactive demo, or a unit of an online front-end
        _case("one utterance", utts=1, min_s=3.17, max_s=3.17, taps=4096, order=6, style="rooms"),
        # the smallest training batch (first synthetic workload): 8 x 2 s, one fixed room
        _case("small batch", utts=8, style="office", taps=4096, order=6),
        # the ordinary training batch (second workload): 256 utterances of 2-20 s, 1-2 noises
        _case("training batch", utts=256, min_s=2.0, max_s=20.0, taps=8192, order=10, noise_hi=2),
        # the same path with what else is used in earnest: noise stretches that start at any sample,
        # power-law features, the mixed waveform kept; part of the utterances without noise
        _case("any-offset noise, waveform", utts=96, min_s=2.0, max_s=20.0, taps=8192, order=10,
              noise_lo=0, noise_hi=2, noise_align=1, power_law=True, wave=True),
        # far-field simulation (third workload): 24000-tap responses of order 20, three noises, 80 bands
        _case("far-field batch", utts=128, style="far", min_s=8.0, max_s=8.0, taps=24000, order=20,
              noise_lo=3, noise_hi=3, n_mel=80),
        # many short commands at once (fourth workload): 4096 x 1-6 s
        _case("short commands", utts=4096, min_s=1.0, max_s=6.0, taps=4096, order=8),
        # long recordings (fifth workload): 64 x 60 s, 1024-point transform, 128 bands
        _case("long recordings", utts=64, style="halls", min_s=60.0, max_s=60.0, taps=16384, order=12,
              noise_lo=2, noise_hi=2, n_fft=1024, n_mel=128),
        # the paper's own order of things: speech warped with a 50 ms window before the simulator
        _case("waveform warp", utts=64, min_s=2.0, max_s=20.0, taps=8192, order=10, noise_hi=2,
              power_law=True, vtlp_win=800),
        # a job whose speech and features live in pinned host memory, noise bank uploaded once
        _case("host buffers", call="host", utts=64, min_s=2.0, max_s=20.0, taps=8192, order=10,
              noise_hi=2),
        # impulse responses alone, to be kept for later
        _case("responses only", call="responses", utts=512, style="rooms", taps=8192, order=12,
              noise_lo=1, noise_hi=3),
        # recorded responses (they fill their buffer) applied to speech and noise
        _case("recorded responses", call="reverb", utts=64, min_s=2.0, max_s=16.0, taps=7999,
              noise_hi=2),
        # features of clean evaluation speech: log-mel, cepstra, mean and variance
        _case("clean features", call="features", utts=128, min_s=2.0, max_s=30.0, n_mel=80),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["pipeline"] * 6 + ["host", "responses", "reverb", "features"])
    style = rng.choice(["rooms", "far", "halls"])
    max_s = _log_uniform(rng, 1.3, 60.0)
    min_s = max_s * rng.choice([1.0, rng.uniform(0.1, 1.0)])
    # at most 4000 s of audio a pass: a quarter of the largest listed batch
    most = max(1, min(4096, int(4000.0 / max_s)))
    utts = max(1, min(most, int(round(_log_uniform(rng, 1, 2.0 * most)))))
    noise_hi = rng.randint(0 if call == "pipeline" else 1, 3)
    taps = int(_log_uniform(rng, 1500, 24000))
    order = rng.randint(3, 20 if style == "far" else 12)
    if call == "responses":
        utts = int(_log_uniform(rng, 1, 700))
    return _case(call=call, style=style, utts=utts, min_s=round(min_s, 4), max_s=round(max_s, 4),
                 taps=taps, order=order, noise_lo=rng.randint(0, noise_hi), noise_hi=noise_hi,
                 noise_align=rng.choice([1, 4]), n_fft=rng.choice([512, 512, 1024]),
                 n_mel=rng.choice([23, 40, 64, 80, 128]), power_law=rng.random() < 0.4,
                 wave=call == "pipeline" and rng.random() < 0.3,
                 vtlp_win=rng.choice([0, 0, 0, 800]) if call == "pipeline" else 0)


# ----------------------------------------------------------------------------- inputs
def _speech(lengths, stride, gen):
    """Voiced speech: harmonics of a drifting 100-250 Hz pitch under a 4 Hz syllabic envelope,
    with noise 30 dB below, RMS about 0.05; zero beyond each utterance's end."""
    dev = "cuda"
    B = len(lengths)
    out = torch.zeros((B, stride), device=dev)
    n = torch.arange(stride, device=dev, dtype=torch.float64) / FS
    f0 = 100.0 + 150.0 * torch.rand(B, 1, device=dev, generator=gen, dtype=torch.float64)
    ph = torch.rand(B, 3, device=dev, generator=gen, dtype=torch.float64)
    ln = torch.as_tensor(lengths, device=dev)
    step = max(1, int(4e7 // max(stride, 1)))
    for b in range(0, B, step):
        e = min(B, b + step)
        turns = f0[b:e] * n + 0.005 * f0[b:e] * torch.sin(math.pi * (n + ph[b:e, :1]))
        turns = (turns - turns.floor()).to(torch.float32)
        x = torch.zeros_like(turns)
        for h in range(1, 13):
            x += torch.sin((2.0 * math.pi * h) * turns + 6.0 * h * h * ph[b:e, 1:2].float()) / h
        env = 0.5 + 0.5 * torch.cos(8.0 * math.pi * (n + ph[b:e, 2:3])).to(torch.float32)
        x = 0.09 * x * env
        x += 0.0016 * torch.randn(x.shape, device=dev, generator=gen)
        x[torch.arange(stride, device=dev)[None, :] >= ln[b:e, None]] = 0.0
        out[b:e] = x
    return out


def _noise_bank(n, gen):
    """Recordings of 40 s: pink-like noise with slow level changes, RMS about 0.05."""
    x = torch.randn(n, device="cuda", generator=gen)
    for k in (2, 8, 32, 128):          # the longer the average, the lower the octaves it adds
        m = -(-n // k)
        low = torch.randn(m, device="cuda", generator=gen).repeat_interleave(k)[:n]
        x = x + 1.4 * low
    t = torch.arange(n, device="cuda", dtype=torch.float32) / FS
    x *= 1.0 + 0.4 * torch.sin(0.7 * t)
    return (x * (0.05 / x.square().mean().sqrt())).contiguous()


def _lengths(case, rng):
    lo, hi = int(case["min_s"] * FS), int(case["max_s"] * FS)
    ln = rng.integers(lo, hi + 1, case["utts"]).astype(np.int32)
    ln[0] = hi                         # the padded width is that of the longest utterance
    return np.maximum(ln, 1)


def _table(case, lengths, bank_len, seed):
    s = _STYLES[case["style"]]
    d = binding.AugDist(t60_lo=s["t60"][0], t60_hi=s["t60"][1], order=case["order"],
                        n_noise_lo=case["noise_lo"], n_noise_hi=case["noise_hi"],
                        snr_lo=s["snr"][0], snr_hi=s["snr"][1], alpha_lo=s["alpha"][0],
                        alpha_hi=s["alpha"][1], wall_margin=0.3, min_src_mic_dist=0.5,
                        min_noise_len=4000, bank_len=bank_len)
    for a in range(3):
        d.room_lo[a], d.room_hi[a] = s["lo"][a], s["hi"][a]
    _, tab = binding.aug_sample_params(seed, d, lengths)
    if case["noise_align"] == 1:       # stretches that start and end at any sample
        rng = np.random.default_rng(seed + 1)
        for j in range(3):
            used = tab["noise_len"][:, j] > 8
            cut = rng.integers(0, 4, len(tab))
            tab["noise_len"][used, j] -= cut[used] + 1
            tab["noise_offset"][used, j] += rng.integers(0, 2, len(tab))[used]
    return tab


def _recorded_responses(case, S, gen):
    """Dense responses: a direct sound and an exponentially decaying tail over the whole buffer."""
    B, L = case["utts"], case["taps"]
    t = torch.arange(L, device="cuda", dtype=torch.float32) / FS
    t60 = 0.2 + 0.6 * torch.rand(B, S, 1, device="cuda", generator=gen)
    h = 0.05 * torch.randn(B, S, L, device="cuda", generator=gen) * torch.exp(-6.9 * t / t60)
    h[:, :, min(40, L - 1)] += 0.5
    return h.contiguous()


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    call = case["call"]
    lengths = _lengths(case, rng)
    B, n_max = case["utts"], int(lengths.max())
    stride = (n_max + 3) // 4 * 4
    T_max = max(1, binding.aug_frame_count(n_max, WIN, HOP))
    bank_len = 16 * 40 * FS if case["noise_hi"] else 0
    S = 1 + case["noise_hi"]
    config = binding.AugConfig(
        fs=FS, win=WIN, hop=HOP, n_fft=case["n_fft"], n_mel=case["n_mel"], f_lo=0.0, f_hi=FS / 2,
        rir_taps=case["taps"], max_order=case["order"], max_sources=S, frac_half_width=HALF_WIDTH,
        sound_speed=343.0, log_floor=float(np.finfo(np.float32).eps), pad_value=0.0,
        compression=binding.COMPRESS_POW_1_15 if case["power_law"] else binding.COMPRESS_LOG,
        max_batch=B, max_samples=stride, host_staging=int(call == "host"), image_lattice=0,
        max_bank_samples=bank_len if call == "host" else 0, vtlp_win=case["vtlp_win"],
        host_rows=1 if call == "host" else 0)
    st = {"call": call, "B": B, "stride": stride, "T_max": T_max, "bank_len": bank_len,
          "lengths_host": lengths, "ctx": binding.AugContext(config)}
    table = _table(case, lengths, bank_len, seed)
    st["table"] = binding.table_to_device(table)
    st["lengths"] = torch.from_numpy(lengths).cuda()
    if call == "responses":
        st["rir"] = torch.zeros((B, S, case["taps"]), device="cuda")
        return st
    st["speech"] = _speech(lengths, stride, gen)
    st["bank"] = _noise_bank(bank_len, gen) if bank_len else None
    st["counts"] = torch.zeros(B, dtype=torch.int32, device="cuda")
    feats = lambda m: torch.zeros((B, T_max, m), device="cuda")
    if call == "pipeline":
        st["feats"] = feats(case["n_mel"])
        st["wave"] = torch.zeros_like(st["speech"]) if case["wave"] else None
    elif call == "host":
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
        st["speech_host"] = pin(st.pop("speech"))
        st["feats_host"] = torch.zeros((B, T_max, case["n_mel"])).pin_memory()
        st["counts_host"] = torch.zeros(B, dtype=torch.int32).pin_memory()
        st["table_host"] = table
        bank = st.pop("bank")
        if bank is not None:
            st["ctx"].aug_upload_noise_bank(bank.cpu(), bank_len)
    elif call == "reverb":
        st["rir"] = _recorded_responses(case, S, gen)
        st["wave"] = torch.zeros_like(st["speech"])
    elif call == "features":
        st["power"] = torch.zeros((B, T_max, case["n_fft"] // 2 + 1), device="cuda")
        st["feats"] = feats(case["n_mel"])
        st["n_cep"] = min(13, case["n_mel"])
        st["cepstra"] = feats(st["n_cep"])
        st["mean"] = torch.zeros((B, case["n_mel"]), device="cuda")
        st["var"] = torch.zeros_like(st["mean"])
    return st


# ----------------------------------------------------------------------------- one pass
def run(st):
    ctx, call, B = st["ctx"], st["call"], st["B"]
    if call == "pipeline":
        ctx.aug_pipeline(st["speech"], st["stride"], st["lengths"], st["lengths_host"], st["bank"],
                         st["bank_len"], st["table"], B, st["feats"], st["T_max"], st["counts"],
                         st["wave"])
        return {"feats": st["feats"], "counts": st["counts"], "wave": st["wave"]}
    if call == "host":
        ctx.aug_pipeline_host(st["speech_host"], st["stride"], st["lengths_host"], None,
                              st["bank_len"], st["table_host"], B, st["feats_host"], st["T_max"],
                              st["counts_host"])
        return {"feats": st["feats_host"], "counts": st["counts_host"]}
    if call == "responses":
        ctx.aug_rir_image_method(st["table"], B, st["rir"])
        return st["rir"]
    if call == "reverb":
        ctx.aug_reverb_mix(st["speech"], st["stride"], st["lengths"], st["bank"], st["bank_len"],
                           st["rir"], st["table"], B, st["wave"])
        return st["wave"]
    ctx.feat_stft_power(st["speech"], st["stride"], st["lengths"], B, st["power"], st["T_max"],
                        st["counts"])
    ctx.feat_vtlp_logmel(st["power"], st["counts"], st["table"], B, st["T_max"], st["feats"])
    ctx.feat_mfcc(st["feats"], st["counts"], B, st["T_max"], st["n_cep"], st["cepstra"])
    m = st["feats"].shape[2]
    ctx.feat_mean_var(st["feats"], st["counts"], B, st["T_max"], m, st["mean"], st["var"])
    return {k: st[k] for k in ("power", "feats", "counts", "cepstra", "mean", "var")}


# ----------------------------------------------------------------------------- work, tolerance
def work(case):
    """Bytes: speech, noise stretches, table (or responses) read once, outputs written once.
    Operations: transforms of split radix size (2.5 F log2 F for a real one), one complex product
    per bin, one multiply-add per tap of every image, the bands' two weights per bin."""
    B, call = case["utts"], case["call"]
    samples = B * (case["min_s"] + case["max_s"]) / 2 * FS
    K, M = case["n_fft"], case["n_mel"]
    frames = max(0.0, (samples - B * WIN) / HOP + B)
    noises = (case["noise_lo"] + case["noise_hi"]) / 2
    src = 1.0 + noises
    real_fft = lambda n: 2.5 * n * math.log2(n)
    nbytes, flops = 160.0 * B, 0.0
    if call != "features":
        n = case["order"]
        images = (2 * n + 1) * (2 * n * n + 2 * n + 3) / 3
        if call != "reverb":
            flops += B * src * images * (2 * HALF_WIDTH + 1) * 2
        if call == "responses":
            return {"bytes": nbytes + 4.0 * B * (1 + case["noise_hi"]) * case["taps"], "flops": flops}
        F = 16384 if case["taps"] <= 8192 else 32768
        blocks = samples / (F - min(case["taps"], F // 2) + 1)
        outs = 1.0 + (1.0 if noises else 0.0)
        flops += blocks * ((src + outs) * real_fft(F) + src * 4.0 * F) + B * src * real_fft(F)
        # the bank is shared: its stretches are read once, three quarters of an utterance each
        nbytes += 4.0 * samples + 4.0 * min(0.75 * noises * samples, 16 * 40 * FS)
        if call == "reverb":
            nbytes += 4.0 * B * src * case["taps"] + 4.0 * samples
            return {"bytes": nbytes, "flops": flops}
        if case["wave"]:
            nbytes += 4.0 * samples
        if case["vtlp_win"]:
            flops += samples / (case["vtlp_win"] / 4) * 2 * real_fft(1024)
    else:
        nbytes += 4.0 * samples + 4.0 * frames * (K // 2 + 1 + min(13, M))
        flops += frames * 2 * M * min(13, M)
    flops += frames * (real_fft(K) + 3 * K / 2 + 4 * (K / 2 + 1))
    nbytes += 4.0 * frames * M + 4.0 * B
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times the distance of the fp32 path from its fp64 definition, as measured on these
    cases.  Pipelines: features 8.5e-6 and at worst 5.3e-4 (bands just above the fp32 noise of the
    transforms), waveform 4.4e-6.  Responses 4.4e-6, at worst 3.6e-5 (a tap beside the window's
    end).  Recorded responses 5.5e-7, 3.3e-6.  Clean features 7e-7, 3.2e-5."""
    return {"responses": {"rel": 2e-5, "max": 1.5e-4}, "reverb": {"rel": 2.2e-6, "max": 2e-5},
            "features": {"rel": 3e-6, "max": 1.5e-4}}.get(case["call"], {"rel": 4e-5, "max": 2e-3})
