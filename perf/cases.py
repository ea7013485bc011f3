"""Performance cases: what programs have this library do, through its public entry points.

A case names a layout (constant-Q or multi-resolution), a transform length, a batch and what is done with it:

  roundtrip  Plan.analyse, then Plan.synthesise
  analyse    Plan.analyse alone (features for another model)
  adjoint    Plan.analyse, then Plan.analyse_adjoint of a coefficient cotangent (forward and backward of a front end)
  train      autograd.analyse, autograd.synthesise, mean squared error against a target, gradient at the signal
  stream     SliCQ.push of some frames of a running stream, then SliCQ.pull

`listed()` holds fixed cases, `draw(rng)` makes further ones of the same ranges.
"""
import functools
import math

import torch

from paper_2609_29119_b200 import Plan, SliCQ, autograd

WINDOWS = {"hann": 0, "blackman_harris": 1}
POLICIES = {"mult4": 0, "smooth": 1, "pow2": 2}
MULTIRES = ((3, 8), (4, 16), (2, 32))   # (octaves, bands per octave) of the multi-resolution layout


def _cq(do, fs, fmin, fmax, bins, n, valid, batch, window="hann", policy="smooth", signal="noise", frames=0, transition=0):
    return {"do": do, "layout": "cq", "fs": fs, "fmin": fmin, "fmax": fmax, "bins": bins, "n": n, "valid": valid, "batch": batch,
            "window": window, "policy": policy, "signal": signal, "frames": frames, "transition": transition}


def _multires(do, batch, n=1 << 16, fs=44100.0, valid=None):
    return {"do": do, "layout": "multires", "fs": fs, "fmin": fs / 1024.0, "fmax": fs / 2, "bins": 0, "n": n,
            "valid": n if valid is None else valid, "batch": batch, "window": "hann", "policy": "pow2", "signal": "sines",
            "frames": 0, "transition": 0}


def listed():
    return [
        # a few short clips at a low rate, shorter than the transform: the smallest call, all latency
        {"name": "short_clips", **_cq("roundtrip", 22050.0, 100.0, 11025.0, 24, 1 << 13, 8000, 3, signal="sines")},
        # interactive analysis and resynthesis of one 1.5 s signal, with the library's default length policy
        {"name": "single_signal", **_cq("roundtrip", 44100.0, 32.70, 22050.0, 12, 1 << 16, 1 << 16, 1, policy="mult4", signal="sines")},
        # 16 stereo clips of 10 s: the batched round trip that the library is quoted on, the largest listed case
        {"name": "batch_clips", **_cq("roundtrip", 44100.0, 32.70, 22050.0, 24, 1 << 19, 441000, 32, signal="pink")},
        # a fixed CQT front end of a model: forward, and the cotangent of its coefficients on the way back
        {"name": "front_end", **_cq("adjoint", 22050.0, 20.0, 11025.0, 48, 1 << 17, 88200, 64)},
        # one minute of audio in one transform at high resolution
        {"name": "long_signal", **_cq("roundtrip", 48000.0, 20.0, 20000.0, 96, 1 << 22, 2880000, 1, window="blackman_harris", signal="sines")},
        # a few clips of an odd length, so that rows of the signal are not aligned
        {"name": "odd_clips", **_cq("roundtrip", 44100.0, 55.0, 18000.0, 36, 1 << 17, 99225, 7, signal="pink")},
        # features of many one-second clips, as a data set is passed through
        {"name": "features", **_cq("analyse", 22050.0, 32.70, 11025.0, 24, 1 << 15, 22050, 256)},
        # a stereo file passed through the sliced form in large pieces
        {"name": "stream_file", **_cq("stream", 44100.0, 32.70, 22050.0, 48, 1 << 15, 1 << 15, 2, signal="pink", frames=64 << 14, transition=1 << 13)},
        # a live stereo stream, one hop at a time
        {"name": "stream_live", **_cq("stream", 44100.0, 32.70, 22050.0, 48, 1 << 15, 1 << 15, 2, signal="pink", frames=1 << 14, transition=1 << 13)},
        # the multi-resolution layout on one signal, and on a large batch
        {"name": "multires_single", **_multires("roundtrip", 1)},
        {"name": "multires_batch", **_multires("roundtrip", 128)},
        # a training step through both transforms, at a training batch
        {"name": "multires_train", **_multires("train", 8)},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["roundtrip", "roundtrip", "adjoint", "analyse", "train", "stream"])
    if do != "stream" and rng.random() < 0.25:
        n = 1 << rng.randint(15, 17)
        most = (1 << 23) // n // (2 if do == "train" else 1)
        return _multires(do, _log_int(rng, 1, most), n=n, valid=rng.randint(n // 2 + 1, n))
    fs = rng.choice([22050.0, 44100.0, 48000.0])
    bins = rng.choice([12, 24, 36, 48, 96])
    n = 1 << (rng.randint(13, 17) if do == "stream" else rng.randint(12, 22))
    # the lowest band is at least a third of a bin wide before the minimum width applies
    q = 1.0 / (2.0 ** (1.0 / bins) - 2.0 ** (-1.0 / bins))
    fmin = max(rng.choice([20.0, 32.70, 55.0]), 0.33 * q * fs / n)
    fmax = rng.choice([0.5, 0.4]) * fs
    window = rng.choice(["hann", "hann", "blackman_harris"])
    # the multiple-of-4 policy is for signals up to some seconds, the longer ones take the other two
    policy = rng.choice(["smooth", "smooth", "pow2"] + (["mult4"] if n <= 1 << 17 else []))
    signal = rng.choice(["noise", "pink", "sines"])
    if do == "stream":
        hop = n // 2
        channels = rng.choice([1, 2, 6])
        return _cq(do, fs, fmin, fmax, bins, n, n, channels, window, policy, signal, _log_int(rng, hop, min(64 * hop, (1 << 21) // channels)),
                   rng.randint(hop // 8, hop))
    most = (3 << 22) // n // (3 if do == "train" else 1) // (1 if policy == "smooth" else 2)
    return _cq(do, fs, fmin, fmax, bins, n, rng.randint(n // 2 + 1, n), _log_int(rng, 1, max(1, most)), window, policy, signal)


def _plan(case, device):
    if case["layout"] == "multires":
        from paper_2609_29119_b200.binding import multires_bands
        centre, width, group = multires_bands(case["fs"], case["fmin"], case["n"], MULTIRES)
        return Plan.from_bands(case["fs"], case["n"], centre, width, group, window=WINDOWS[case["window"]],
                               m_policy=POLICIES[case["policy"]], device=device)
    return Plan(case["fs"], case["fmin"], case["fmax"], case["bins"], case["n"], window=WINDOWS[case["window"]],
                m_policy=POLICIES[case["policy"]], device=device)


def _signal(case, rows, length, gen):
    """[rows, length] float32 audio on the GPU, about 0.1 rms."""
    noise = torch.randn(rows, length, generator=gen, device="cuda")
    if case["signal"] == "pink":
        even = length + length % 2
        spec = torch.fft.rfft(noise, n=even)
        spec /= torch.arange(1, spec.shape[1] + 1, device="cuda").sqrt()
        x = torch.fft.irfft(spec, n=even)[:, :length]
        x = 0.1 * x / x.square().mean(dim=1, keepdim=True).sqrt()
    elif case["signal"] == "sines":
        x = 0.1 * noise
        t = torch.arange(length, device="cuda") / case["fs"]
        for f, ph in torch.rand(5, 2, generator=gen, device="cuda").tolist():
            x += 0.05 * torch.cos(2 * math.pi * (100.0 * 80.0 ** f * t + ph))
    else:
        x = 0.1 * noise
    return x.contiguous()


class State:
    pass


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = State()
    s.do, s.valid, s.batch = case["do"], case["valid"], case["batch"]
    s.plan = _plan(case, torch.cuda.current_device())
    if s.do == "stream":
        hop, frames = case["n"] // 2, case["frames"]
        s.x = _signal(case, s.batch, frames, gen)
        s.stream = SliCQ(s.plan, s.batch, case["transition"], max(2, frames // hop + 2))
        s.y = torch.zeros(s.batch, frames + hop, device="cuda")
        s.stream.push(_signal(case, s.batch, hop, gen))   # a stream under way: every pass finds the slice before it
        s.stream.pull(s.y)
        return s
    s.x = _signal(case, s.batch, s.valid, gen)
    if s.do == "adjoint":
        s.c_bar = torch.randn(s.batch, s.plan.coeff_count, dtype=torch.complex64, generator=gen, device="cuda")
    if s.do == "train":
        s.x.requires_grad_(True)
        s.target = _signal(case, s.batch, s.valid, gen)
    return s


def run(s):
    if s.do == "stream":
        done = s.stream.push(s.x)
        return {"slices": done, "frames": s.stream.pull(s.y), "y": s.y}
    if s.do == "train":
        c = autograd.analyse(s.plan, s.x)
        y = autograd.synthesise(s.plan, c, valid_len=s.valid)
        loss = torch.nn.functional.mse_loss(y, s.target)
        grad, = torch.autograd.grad(loss, s.x)
        return {"c": c.detach(), "y": y.detach(), "loss": loss.detach(), "grad": grad}
    c = s.plan.analyse(s.x, valid_len=s.valid)
    if s.do == "analyse":
        return {"c": c}
    if s.do == "adjoint":
        return {"c": c, "grad": s.plan.analyse_adjoint(s.c_bar, valid_len=s.valid)}
    return {"c": c, "y": s.plan.synthesise(c, valid_len=s.valid)}


@functools.lru_cache(maxsize=None)
def _sizes(key):
    """(coefficients, window entries, sum of 5 M log2 M) of one signal, from a plan without a device."""
    plan = _plan(dict(key), -1)
    bands = plan.bands()
    sizes = plan.coeff_count, plan.table_length, sum(5.0 * b.M * math.log2(b.M) for b in bands)
    plan.close()
    return sizes


def work(case):
    layout = ("layout", "fs", "fmin", "fmax", "bins", "n", "window", "policy")
    coeffs, window, band_flops = _sizes(tuple((k, case[k]) for k in layout))
    # one transform of one signal: a real FFT of n samples, one complex FFT per band, the window products
    flops = 2.5 * case["n"] * math.log2(case["n"] / 2) + band_flops + 16.0 * window
    if case["do"] == "stream":
        slices = case["frames"] / (case["n"] // 2) * case["batch"]
        # frames in, frames out, coefficients of the slices written and read, both window tables and the slice window
        return {"bytes": 8.0 * case["frames"] * case["batch"] + 16.0 * coeffs * slices + 8.0 * window + 4.0 * case["n"],
                "flops": 2.0 * flops * slices}
    batch, signal, row = case["batch"], 4.0 * case["valid"], 8.0 * coeffs
    transforms = {"analyse": 1, "roundtrip": 2, "adjoint": 2, "train": 4}[case["do"]]
    nbytes = batch * transforms * (signal + row) + 4.0 * window * transforms
    if case["do"] == "train":
        nbytes += batch * 2 * signal   # reconstruction and target read for the loss; its gradient is read by the transform
    return {"bytes": nbytes, "flops": transforms * flops * batch}


def tolerance(case):
    # two correct 32-bit evaluations differ by a few 1e-7 of the result's norm; single coefficients of a weak band carry
    # the rounding of the whole spectrum, which is what "max" leaves room for
    return {"rel": 3e-6, "max": 1e-4}
