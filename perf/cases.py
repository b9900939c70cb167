"""Performance cases of the CWT library: what its users have it compute, through its public entry points.

Sizes come from the repository's workloads (eeg_synth.workload, bench.py), its length sweep and its tests.
Signals are synthetic EEG: band sinusoids of 5-30 uV, 1/f noise and white noise, drawn on the GPU from the seed.

The phase output is not among the cases: it jumps by 2 pi where it crosses the branch cut and is arbitrary where
the coefficient vanishes, so two correct results cannot be compared value by value.  It follows from the complex
output, which is here.
"""
import math

import numpy as np
import torch

from paper_2506_07793_gb300 import cwt

WINDOW = 2048  # samples of a live stream's window (the server's only size)


def listed():
    return [
        # one second of an 8-channel headset at 500 Hz in double precision: the smallest call, once per second
        dict(name="second_f64", path="plan", channels=8, samples=500, fs=500.0, scales=40, f_lo=1.0, f_hi=40.0,
             log=False, c_lo=7.0, c_hi=7.0, outputs="power", dtype="f64", pad="pow2", edge="cyclic",
             wavelet="morlet", decimation=1, precision="fp32"),
        # a brain-computer-interface loop that may not allocate: two seconds of 16 channels, every call
        dict(name="loop_noalloc", path="noalloc", channels=16, samples=2000, fs=1000.0, scales=40, f_lo=4.0,
             f_hi=90.0, log=True, c_lo=3.0, c_hi=7.0, outputs="complex+power"),
        # one trial of the paper's length sweep, a prime length: gamma band, complex coefficients
        dict(name="trial_1009", path="plan", channels=64, samples=1009, fs=1000.0, scales=61, f_lo=30.0, f_hi=90.0,
             log=False, c_lo=7.0, c_hi=7.0, outputs="complex", dtype="f32", pad="pow2", edge="cyclic",
             wavelet="morlet", decimation=1, precision="fp32"),
        # a ragged trial under the paper's padding: 3001 samples pad to 3024, no round number of seconds
        dict(name="trial_3001_smooth", path="plan", channels=64, samples=3001, fs=1000.0, scales=61, f_lo=2.0,
             f_hi=90.0, log=True, c_lo=3.0, c_hi=10.0, outputs="complex+power", dtype="f32", pad="smooth",
             edge="cyclic", wavelet="morlet", decimation=1, precision="fp32"),
        # generalized Morse wavelets, power kept at every 4th sample (a time-frequency map to look at)
        dict(name="morse_decimated", path="plan", channels=64, samples=8000, fs=500.0, scales=80, f_lo=2.0,
             f_hi=100.0, log=True, c_lo=17.5, c_hi=17.5, outputs="power", dtype="f32", pad="pow2", edge="cyclic",
             wavelet="gmw", decimation=4, precision="fp32"),
        # the headline workload: ten seconds of 64 channels, 100 scales, under the paper's padding ...
        dict(name="ten_seconds", path="plan", channels=64, samples=10000, fs=1000.0, scales=100, f_lo=1.0,
             f_hi=100.0, log=True, c_lo=3.0, c_hi=10.0, outputs="complex+power", dtype="f32", pad="smooth",
             edge="cyclic", wavelet="morlet", decimation=1, precision="fp32"),
        # ... and under the library's default power-of-two padding
        dict(name="ten_seconds_pow2", path="plan", channels=64, samples=10000, fs=1000.0, scales=100, f_lo=1.0,
             f_hi=100.0, log=True, c_lo=3.0, c_hi=10.0, outputs="complex+power", dtype="f32", pad="pow2",
             edge="cyclic", wavelet="morlet", decimation=1, precision="fp32"),
        # half a minute of 16 channels on the tensor-core inverse FFTs that a plan may ask for
        dict(name="half_minute_tc", path="plan", channels=16, samples=30000, fs=1000.0, scales=64, f_lo=1.0,
             f_hi=100.0, log=True, c_lo=7.0, c_hi=7.0, outputs="power", dtype="f32", pad="pow2", edge="cyclic",
             wavelet="morlet", decimation=1, precision="tc_fp16"),
        # a minute of 8 channels at 1 kHz with linear edges under the paper's padding
        dict(name="minute_linear", path="plan", channels=8, samples=60000, fs=1000.0, scales=100, f_lo=1.0,
             f_hi=100.0, log=True, c_lo=3.0, c_hi=10.0, outputs="complex+power", dtype="f32", pad="smooth",
             edge="linear", wavelet="morlet", decimation=1, precision="fp32"),
        # a minute at 2048 Hz, 32 channels of the precision workload: the longest rows, the largest output
        dict(name="minute_2048", path="plan", channels=32, samples=122880, fs=2048.0, scales=128, f_lo=0.5,
             f_hi=200.0, log=True, c_lo=7.0, c_hi=7.0, outputs="power", dtype="f32", pad="pow2", edge="cyclic",
             wavelet="morlet", decimation=1, precision="fp32"),
        # event-locked epochs of uneven length in one call: an eighth of the batching workload
        dict(name="epochs_256", path="batch", epochs=256, channels=64, n_lo=256, n_hi=8192, fs=1000.0, scales=64,
             f_lo=2.0, f_hi=80.0, c_lo=3.0, c_hi=12.0, decimation=4, outputs="power"),
        # live recordings: one 50 ms hop of each of 16 streams (8-128 channels, 250-4000 Hz), pushed, stepped, pulled
        dict(name="live_16", path="live", streams=16, scales=64, f_lo=1.0, f_hi=100.0, cycles=7.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "plan", "plan", "plan", "long", "tc", "f64", "noalloc", "batch", "live"])
    if kind == "live":
        return dict(path="live", streams=rng.randint(1, 16), scales=rng.randint(16, 64), f_lo=rng.uniform(1.0, 4.0),
                    f_hi=rng.uniform(40.0, 110.0), cycles=rng.uniform(4.0, 7.0))
    if kind == "batch":
        n_lo = _log_int(rng, 200, 1500)
        n_hi, scales, d = _log_int(rng, 2 * n_lo, 8192), rng.randint(20, 64), rng.choice([1, 2, 4, 4, 5])
        channels = rng.choice([8, 19, 32, 64])
        epochs = min(_log_int(rng, 8, 250), int(8e8 * d / (channels * scales * (n_lo + n_hi) / 2 * max(1, 4 / d))))
        return dict(path="batch", epochs=epochs, channels=channels, n_lo=n_lo, n_hi=n_hi, fs=1000.0, scales=scales,
                    f_lo=rng.uniform(5.0, 15.0), f_hi=rng.uniform(60.0, 100.0), c_lo=3.0, c_hi=rng.uniform(7.0, 12.0),
                    decimation=d, outputs="power")
    fs = rng.choice([250.0, 500.0, 512.0, 1000.0, 1000.0, 2048.0])
    lo, hi = dict(plan=(100, 16000), long=(16400, 120000), tc=(8200, 60000), f64=(100, 2500), noalloc=(100, 8000))[kind]
    n = _log_int(rng, lo, hi)
    f_lo = max(rng.uniform(0.5, 4.0), 3.0 * fs / n)
    f_hi = min(max(rng.uniform(40.0, 120.0), 2.5 * f_lo), 0.4 * fs)
    f_lo = min(f_lo, 0.5 * f_hi)
    scales = rng.randint(20, 128)
    most = 1.5e8 if kind == "long" else 6e7 if kind != "noalloc" else 2e6  # coefficients of one call
    if kind == "noalloc":
        scales = min(scales, 50)
    channels = max(1, min(_log_int(rng, 4, 256), int(most / (scales * n))))
    case = dict(path="plan", channels=channels, samples=n, fs=fs, scales=scales, f_lo=f_lo, f_hi=f_hi, log=True,
                c_lo=rng.uniform(3.0, 7.0), c_hi=rng.uniform(7.0, 12.0),
                outputs=rng.choice(["power", "complex", "complex+power"]))
    if kind == "noalloc":
        return dict(case, path="noalloc")
    case.update(dtype="f64" if kind == "f64" else "f32", pad=rng.choice(["pow2", "smooth"]), edge="cyclic",
                wavelet="morlet", decimation=1, precision="fp32")
    if kind == "tc":
        case.update(pad="pow2", precision=rng.choice(["tc_fp16", "tc_bf16"]))
    elif kind in ("plan", "long"):
        case.update(edge=rng.choice(["cyclic", "cyclic", "linear"]), decimation=rng.choice([1, 1, 1, 2, 3, 4, 8]))
        if case["edge"] == "cyclic" and rng.random() < 0.25:
            case.update(wavelet="gmw", c_lo=rng.uniform(8.0, 20.0), c_hi=20.0)
        if kind == "long" and case["edge"] == "linear":  # room for the widest wavelet's support
            case["samples"] = min(n, 90000)
            case["f_lo"] = max(case["f_lo"], 2.0)
    return case


# ---- inputs -----------------------------------------------------------------------------------------------------

def _device():
    return torch.device("cuda")


def _eeg(channels, n, fs, seed):
    """[channels][n] float64 synthetic EEG in microvolts on the GPU."""
    g = torch.Generator(device=_device())
    g.manual_seed(1_000_003 * int(seed) + 17)
    opt = dict(generator=g, device=_device(), dtype=torch.float64)
    t = torch.arange(n, device=_device(), dtype=torch.float64) / fs
    x = 2.0 * torch.randn(channels, n, **opt)
    for centre in (2.0, 6.0, 10.0, 20.0, 40.0):
        f = centre * (0.9 + 0.2 * torch.rand(channels, 1, **opt))
        amp = 5.0 + 25.0 * torch.rand(channels, 1, **opt)
        x += amp * torch.cos(2.0 * math.pi * (f * t + torch.rand(channels, 1, **opt)))
    white = torch.fft.rfft(torch.randn(channels, n, **opt))
    k = torch.arange(white.shape[1], device=_device(), dtype=torch.float64)
    pink = torch.fft.irfft(white * torch.where(k > 0, k.clamp(min=1.0).rsqrt(), 0.0 * k), n=n)
    return x + 10.0 * pink / pink.square().mean(dim=1, keepdim=True).sqrt()


def _scales(case):
    S = case["scales"]
    if case.get("log", True):
        f = np.geomspace(case["f_lo"], case["f_hi"], S)
    else:
        f = np.linspace(case["f_lo"], case["f_hi"], S)
    if case["path"] == "live":
        return f, np.full(S, float(case["cycles"]))
    if case["path"] == "batch":
        return f, np.clip(f / 2.0, case["c_lo"], case["c_hi"])
    return f, np.linspace(case["c_lo"], case["c_hi"], S)


def _signal(case, seed):
    x = _eeg(case["channels"], case["samples"], case["fs"], seed)
    return x if case.get("dtype") == "f64" else x.float()


def _epochs(case, seed):
    """(lengths, packed float32 input): windows of one continuous recording.  The lengths are the case's own, the
    recording and the windows' places in it the seed's."""
    lengths = np.random.default_rng([case["n_lo"], case["n_hi"]]).integers(case["n_lo"], case["n_hi"] + 1,
                                                                          size=case["epochs"])
    rng = np.random.default_rng([int(seed), 3])
    rec = _eeg(case["channels"], 1 << 17, case["fs"], seed).float()
    starts = rng.integers(0, rec.shape[1] - lengths + 1)
    return lengths, torch.cat([rec[:, s:s + n].reshape(-1) for s, n in zip(starts.tolist(), lengths.tolist())])


def _stream_specs(case):
    chans, rates = (8, 32, 64, 128, 32), (250.0, 500.0, 1000.0, 2000.0, 4000.0, 1000.0, 500.0)
    return [(chans[i % 5], rates[i % 7]) for i in range(case["streams"])]


class _Live:
    """A server with its open streams and the recordings that are fed to them."""

    def __init__(self, case, seed):
        f, c = _scales(case)
        self.server = cwt.cwt_server_create(f, c)
        self.streams = []
        for i, (channels, fs) in enumerate(_stream_specs(case)):
            hop = math.ceil(fs * 0.05 - 1e-9)
            hops = -(-WINDOW // hop) + 8
            rec = _live_recording(case, seed, i, channels, hops * hop, fs)
            blocks = [np.ascontiguousarray(rec[:, k * hop:(k + 1) * hop]) for k in range(hops)]
            out = np.empty((1, channels, case["scales"], hop), dtype=np.float32)
            self.streams.append(dict(id=cwt.cwt_stream_open(self.server, channels, fs), blocks=blocks, out=out, at=0))
        behind = [len(s["blocks"]) - 8 for s in self.streams]  # a full window before the first timed hop
        while any(s["at"] < b for s, b in zip(self.streams, behind)):
            for s, b in zip(self.streams, behind):
                for _ in range(min(8, b - s["at"])):
                    self.push(s)
            cwt.cwt_server_step(self.server)
            cwt.cwt_server_sync(self.server)
            for s in self.streams:
                while cwt.cwt_stream_pull(self.server, s["id"], s["out"])[0]:
                    pass

    def push(self, s):
        cwt.cwt_stream_push(self.server, s["id"], s["blocks"][s["at"] % len(s["blocks"])])
        s["at"] += 1

    def __del__(self):
        cwt.cwt_server_destroy(self.server)


def _live_recording(case, seed, i, channels, n, fs):
    return _eeg(channels, n, fs, 100 * int(seed) + i).float().cpu().numpy()


def prepare(case, seed):
    f, c = _scales(case)
    path = case["path"]
    if path == "live":
        return dict(path=path, live=_Live(case, seed))
    kinds = case["outputs"].split("+")
    if path == "noalloc":
        x = _signal(case, seed)
        shape = (case["channels"], case["scales"], case["samples"])
        out = {k: torch.empty(shape, dtype=torch.complex64 if k == "complex" else torch.float32, device=x.device)
               for k in kinds}
        return dict(path=path, x=x, out=out, fs=case["fs"], f=f, c=c)
    if path == "batch":
        lengths, x = _epochs(case, seed)
        plan = cwt.CWT(case["channels"], case["n_hi"], case["fs"], f, c, outputs=("power",),
                       decimation=case["decimation"])
        epochs, n_in, n_out = cwt.pack_epochs(lengths, case["channels"], case["scales"], case["decimation"])
        return dict(path=path, plan=plan, epochs=epochs, x=x,
                    out=torch.empty(n_out, dtype=torch.float32, device=x.device))
    plan = cwt.CWT(case["channels"], case["samples"], case["fs"], f, c, outputs=tuple(kinds),
                   wavelet=case["wavelet"], dtype=case["dtype"], decimation=case["decimation"], pad=case["pad"],
                   edge=case["edge"], precision=case["precision"])
    x = _signal(case, seed)
    return dict(path=path, plan=plan, x=x, out=plan.alloc_outputs(x.device))


def run(state):
    path = state["path"]
    if path == "plan":
        return state["plan"](state["x"], out=state["out"])
    if path == "batch":
        cwt.cwt_execute_batch(state["plan"].plan, state["epochs"], state["x"], power_out=state["out"])
        return state["out"]
    if path == "noalloc":
        x, out = state["x"], state["out"]
        cwt.cwt_execute_noalloc(x, x.shape[0], x.shape[1], state["fs"], state["f"], state["c"],
                                complex_out=out.get("complex"), power_out=out.get("power"))
        return out
    live = state["live"]
    for s in live.streams:
        live.push(s)
    cwt.cwt_server_step(live.server)
    cwt.cwt_server_sync(live.server)
    for s in live.streams:
        cwt.cwt_stream_pull(live.server, s["id"], s["out"])
    return [s["out"] for s in live.streams]


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def work(case):
    """Bytes: the signal read and the requested outputs written once.  Operations: a real forward FFT per channel
    and, per output coefficient, an inverse transform from the bins that the scale's wavelet occupies (those above
    1e-10 of its peak), 5 log2 of their count."""
    f, c = _scales(case)

    def one(channels, n, n_out, fs, per_in, per_out):
        bins = np.maximum(2.0, np.minimum(13.6 * f / c * n / fs, n))
        flops = channels * (2.5 * n * math.log2(max(n, 2)) + float(np.sum(5.0 * n_out * np.log2(bins))))
        return channels * (n * per_in + len(f) * n_out * per_out), flops

    if case["path"] == "live":
        parts = []
        for channels, fs in _stream_specs(case):
            hop = math.ceil(fs * 0.05 - 1e-9)
            parts.append(one(channels, WINDOW, hop, fs, 4, 4))
    elif case["path"] == "batch":
        mean = (case["n_lo"] + case["n_hi"]) / 2
        b, w = one(case["channels"], mean, mean / case["decimation"], case["fs"], 4, 4)
        parts = [(case["epochs"] * b, case["epochs"] * w)]
    else:
        size = 8 if case.get("dtype") == "f64" else 4
        per_out = sum(2 * size if k == "complex" else size for k in case["outputs"].split("+"))
        n = case["samples"]
        parts = [one(case["channels"], n, -(-n // case.get("decimation", 1)), case["fs"], size, per_out)]
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


# ---- the same values in 64 bits -----------------------------------------------------------------------------------

def _spectrum(wavelet, f, c, fs, N):
    """[S][N] float64: the unit-energy wavelets' spectra on the N bins, every alias summed."""
    nu0 = np.arange(N) / N * fs
    W = np.zeros((len(f), N))
    for s in range(len(f)):
        F, sg = f[s], c[s]
        if wavelet == "gmw":
            beta, gamma = sg, 3.0
            wp = (beta / gamma) ** (1.0 / gamma)
            la = math.log(2.0) + beta / gamma * (1.0 + math.log(gamma) - math.log(beta))
            for q in range(0, 2 + int(12.0 * F / fs)):
                w = wp * (nu0 + q * fs) / F
                with np.errstate(divide="ignore"):
                    W[s] += np.exp(la + beta * np.log(w) - w ** gamma)
        else:
            reach, kappa = 40.0 * F / sg, math.exp(-0.5 * sg * sg)
            for q in range(math.floor(-reach / fs) - 1, math.ceil((F + reach) / fs) + 1):
                u = (nu0 + q * fs) / F
                W[s] += np.exp(-0.5 * sg * sg * (u - 1.0) ** 2) - kappa * np.exp(-0.5 * sg * sg * u * u)
    return torch.from_numpy(W / np.sqrt((W * W).sum(axis=1, keepdims=True) / N)).to(_device())


def _padded(n, pad):
    """The padded length: the next power of two, or the next 2,3,5,7-smooth length (None where the library may pass
    over it: 3^10, 5^7 and some above 84000)."""
    m = max(n, 32)
    if pad == "pow2":
        return 1 << (m - 1).bit_length()
    while True:
        rest = m
        for p in (2, 3, 5, 7):
            while rest % p == 0:
                rest //= p
        if rest == 1:
            return None if m in (59049, 78125) or m > 84000 else m
        m += 1


def _exact_rows(x, W, kinds, n_keep, first, step, out):
    """Fills out[kind][channel] with the transform of the float64 rows x, kept at [first, first + n_keep) by step."""
    N = W.shape[1]
    for ch in range(x.shape[0]):
        z = torch.fft.ifft(torch.fft.fft(x[ch], n=N) * W, dim=1)[:, first:first + n_keep:step]
        for k in kinds:
            out[k][ch] = z if k == "complex" else z.real.square() + z.imag.square()


def exact(case, seed):
    f, c = _scales(case)
    path = case["path"]
    if path == "live":
        got = []
        for i, (channels, fs) in enumerate(_stream_specs(case)):
            hop = math.ceil(fs * 0.05 - 1e-9)
            hops = -(-WINDOW // hop) + 8
            rec = torch.from_numpy(_live_recording(case, seed, i, channels, hops * hop, fs)).to(_device()).double()
            end = (hops - 7) * hop
            out = torch.empty(1, channels, len(f), hop, dtype=torch.float64, device=_device())
            lo = WINDOW - (WINDOW - hop) // 2 - hop
            _exact_rows(rec[:, end - WINDOW:end], _spectrum("morlet", f, c, fs, WINDOW), ["power"], hop, lo, 1,
                        {"power": out[0]})
            got.append(out.cpu().numpy())
        return got
    kinds = case["outputs"].split("+")
    if path == "batch":
        lengths, x = _epochs(case, seed)
        C, d, at, parts, spectra = case["channels"], case["decimation"], 0, [], {}
        for n in lengths.tolist():
            N = _padded(n, "pow2")
            if N not in spectra:
                spectra[N] = _spectrum("morlet", f, c, case["fs"], N)
            out = torch.empty(C, len(f), -(-n // d), dtype=torch.float64, device=_device())
            _exact_rows(x[at:at + C * n].reshape(C, n).double(), spectra[N], kinds, n, 0, d, {"power": out})
            at += C * n
            parts.append(out.reshape(-1))
        return torch.cat(parts)
    n, d = case["samples"], case.get("decimation", 1)
    extra = 0
    if case.get("edge") == "linear":  # room for the widest wavelet: 6.5 standard deviations of its envelope
        extra = 1 + max(math.ceil(6.5 * b / (2.0 * math.pi * a) * case["fs"]) for a, b in zip(f, c))
    N = _padded(n + extra, case.get("pad", "pow2"))
    if N is None:
        return None
    shape = (case["channels"], len(f), -(-n // d))
    out = {k: torch.empty(shape, dtype=torch.complex128 if k == "complex" else torch.float64, device=_device())
           for k in kinds}
    _exact_rows(_signal(case, seed).double(), _spectrum(case.get("wavelet", "morlet"), f, c, case["fs"], N), kinds, n,
                0, d, out)
    return out
