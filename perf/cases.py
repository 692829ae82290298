"""The work that a user of the readout library has it do, as measurable cases.

Every case goes through the Python binding's public calls (``Plan.push_into``,
``Batch.push``, ``Tx.synthesize``): a program keeps a plan (or a batch, or a
transmit generator) with its output buffers and hands it one buffer of the
radio's stream per call.  A streaming plan continues its stream from call to
call; ``exact`` gives the frames of the first call on a new plan.

Sizes are those of the repository's workloads and tests: the 64-channel filter
bank of 2^20 samples, the 4096-channel one at the paper's rate, Fig. 3's 10^5
channels, the 2048-tone demodulation, the mixed streams of the batched and
serving workloads (N in {256, 1024, 4096, 16384}, T in {4, 8, 16}; 64 to 4096
tones, L in {1024, 4096}, D in {512, 2048}; buffers from 1 MB on), the chirped
readout and the transmit comb.
"""
import math

import numpy as np
import torch

from paper_1812_02200_gb300 import rfr

DEV = "cuda:0"
FULL_SCALE = 8191                     # 14-bit ADC
LOWPASS = 40e3 / 200e6                # demodulation: 40 kHz at 200 Ms/s


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one short capture on a coarse filter bank: 2^20 samples, 64 channels
        dict(name="pfb_64_short", kind="pfb", N=64, T=4, hop=64, window="hann", beta=0.0, tones=16, full=True,
             n=1 << 20),
        # the smallest streaming call: one 1 MB radio buffer, where launches and latency count
        dict(name="pfb_4096_buffer", kind="pfb", N=4096, T=8, hop=4096, window="kaiser", beta=9.0, tones=1000,
             full=True, n=1 << 18),
        # a radio whose buffers are no multiple of anything; only the tones are kept
        dict(name="pfb_4096_ragged", kind="pfb", N=4096, T=8, hop=4096, window="kaiser", beta=9.0, tones=1000,
             full=False, n=3000001),
        # 1.3 s of a 200 Ms/s stream at once: spectrum and 1000 tones
        dict(name="pfb_4096_capture", kind="pfb", N=4096, T=8, hop=4096, window="kaiser", beta=9.0, tones=1000,
             full=True, n=1 << 28),
        # fine channels of the mixed streams
        dict(name="pfb_16384", kind="pfb", N=16384, T=8, hop=16384, window="kaiser", beta=9.0, tones=1000,
             full=True, n=1 << 26),
        # Fig. 3's channel count (no power of two), the paper's Hamming window
        dict(name="pfb_100000", kind="pfb", N=100000, T=4, hop=100000, window="hamming", beta=0.0, tones=1000,
             full=True, n=1 << 27),
        # oversampled four times
        dict(name="pfb_4096_oversampled", kind="pfb", N=4096, T=8, hop=1024, window="kaiser", beta=9.0, tones=1000,
             full=True, n=1 << 26),
        # direct demodulation of a full comb over 0.67 s
        dict(name="demod_2048", kind="demod", tones=2048, L=4096, D=2048, n=1 << 27),
        # direct demodulation of one odd-sized 4 MB radio buffer
        dict(name="demod_300_buffer", kind="demod", tones=300, L=1024, D=512, n=1000003),
        # chirped readout: the stream against 8 chirps
        dict(name="chirp_8", kind="chirp", tones=8, L=4096, D=2048, n=1 << 24),
        # 21 ms of the transmit comb
        dict(name="tx_1000", kind="tx", tones=1000, n=1 << 22),
        # 24 mixed readouts advanced together (the batched workload of the benchmark)
        dict(name="batch_24", kind="batch", streams=24, lo=22.0, hi=26.0,
             spec_seed=1812022004),
    ]


def _log_int(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(lo, hi)))


def draw(rng):
    kind = rng.choice(["pfb", "pfb", "pfb", "anyn", "over", "demod", "demod", "demod", "chirp", "tx", "batch"])
    if kind in ("pfb", "anyn", "over"):
        hop = None
        if kind == "pfb":
            N, T = rng.choice([64, 256, 1024, 4096, 4096, 16384]), rng.choice([4, 8, 16])
            n = _log_int(rng, 18, 27)
        elif kind == "anyn":
            N, T = rng.choice([1000, 10000, 100000, 1000000]), rng.choice([4, 8])
            n = _log_int(rng, 23, 26)
        else:
            N, T = 4096, 8
            hop = rng.choice([1024, 2048])
            n = _log_int(rng, 18, 25.5)
        if rng.random() < 0.5:
            n -= n % 1024
        window = rng.choice(["hann", "hamming", "kaiser"])
        return dict(kind="pfb", N=N, T=T, hop=hop or N, window=window, beta=9.0 if window == "kaiser" else 0.0,
                    tones=max(1, min(N // 4, _log_int(rng, 4, 10))), full=rng.random() < 0.6, n=n)
    if kind == "demod":
        c = dict(kind="demod", tones=_log_int(rng, 6, 12), L=rng.choice([1024, 4096]), D=rng.choice([512, 2048]))
        n = min(_log_int(rng, 18, 25), (1 << 39) // (c["tones"] * c["L"] // c["D"]))    # no more than the listed one
        return dict(c, n=n - n % 1024 if rng.random() < 0.5 else n)
    if kind == "chirp":
        return dict(kind="chirp", tones=rng.randint(1, 16), L=rng.choice([1024, 4096]), D=2048, n=_log_int(rng, 18, 24))
    if kind == "tx":
        return dict(kind="tx", tones=_log_int(rng, 6, 9.9), n=_log_int(rng, 18, 22))
    return dict(kind="batch", streams=rng.randint(3, 16), lo=18.0, hi=24.0, spec_seed=rng.randint(0, 1 << 30))


def _streams(case):
    """The streams of a batch: half filter banks, half demodulations."""
    r = np.random.default_rng(case["spec_seed"])
    out = []
    for _ in range(case["streams"]):
        n = int(round(2.0 ** r.uniform(case["lo"], case["hi"])))
        n -= n % 1024
        if r.uniform() < 0.5:
            N, T = int(r.choice([256, 1024, 4096, 16384])), int(r.choice([4, 8, 16]))
            out.append(dict(kind="pfb", N=N, T=T, hop=N, window="kaiser", beta=9.0, tones=min(1000, N // 4), full=True,
                            n=n))
        else:
            tones = int(round(2.0 ** r.uniform(6.0, 12.0)))
            out.append(dict(kind="demod", tones=tones, L=int(r.choice([1024, 4096])), D=int(r.choice([512, 2048])),
                            n=n))
    return out


# ----------------------------------------------------------------- inputs
def _rngs(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return np.random.default_rng(seed), g


def _turns(phase):
    """exp(i 2 pi phase / 2^64) of int64 phases, in 64 bits."""
    a = phase.to(torch.float64) * (math.pi / 2.0 ** 63)
    return torch.complex(torch.cos(a), torch.sin(a))


def _quantise(x, a, z, sigma, g):
    v = torch.view_as_real(z)
    v = v + sigma * torch.randn(v.shape, generator=g, device=DEV)
    x[a:a + z.shape[0]] = v.round_().clamp_(-FULL_SCALE - 1, FULL_SCALE).to(torch.int16)


def _signal(case, seed):
    """Tone words and the stream: a comb plus noise, rounded to the ADC's 14 bits."""
    r, g = _rngs(seed)
    n, nt = case["n"], case["tones"]
    x = torch.empty((n, 2), dtype=torch.int16, device=DEV)
    if case["kind"] == "pfb":
        # tones at random bin centres, no two in one bin; the comb repeats every N samples
        N = case["N"]
        bins = r.permutation(N)[:nt]
        words = np.array([((int(b) << 64) + N // 2) // N % 2 ** 64 for b in bins], np.uint64)
        u = r.uniform(0.5, 1.0, nt)
        coef = u * (FULL_SCALE - 16.0) / u.sum() * np.exp(2j * np.pi * r.uniform(0, 1, nt))
        spec = torch.zeros(N, dtype=torch.complex128, device=DEV)
        spec[torch.from_numpy(bins).to(DEV)] = torch.from_numpy(coef).to(DEV)
        one = (torch.fft.ifft(spec) * N).to(torch.complex64)
        step = max(1, (1 << 24) // N)
        blk = one.repeat(step)
        for a in range(0, n, step * N):
            _quantise(x, a, blk[:n - a], 4.0, g)
        return words, x
    # tones anywhere (off-bin); the comb's RMS is an eighth of full scale or so
    words = r.integers(0, 2 ** 64 - 1, size=nt, dtype=np.uint64, endpoint=True)
    amp = r.uniform(100.0, 1000.0, nt)
    amp *= math.sqrt(((FULL_SCALE / 6.0) ** 2 - 64.0) / (0.5 * float(np.sum(amp * amp))))
    coef = torch.from_numpy(amp * np.exp(2j * np.pi * r.uniform(0, 1, nt))).to(DEV)
    w = torch.from_numpy(words.view(np.int64)).to(DEV)
    B = 4096
    e = _turns(w[:, None] * torch.arange(B, device=DEV)[None, :]).to(torch.complex64)
    for a in range(0, n, 1024 * B):
        q = torch.arange(a, min(n, a + 1024 * B), B, device=DEV)
        z = ((_turns(q[:, None] * w[None, :]) * coef[None, :]).to(torch.complex64) @ e).reshape(-1)
        _quantise(x, a, z[:n - a], 8.0, g)
    return words, x


def _chirps(case, seed):
    """Start and rate words of upward chirps that cross the band in about 20 ms."""
    r = np.random.default_rng(seed + 1)
    start = r.integers(0, 2 ** 64 - 1, size=case["tones"], dtype=np.uint64, endpoint=True)
    rate = np.array([int(2 ** 64 * k / 200e6) for k in r.uniform(20.0, 60.0, case["tones"])], np.uint64)
    return start, rate


def _make(case, seed):
    """A plan, its input and its output buffers."""
    words, x = _signal(case, seed)
    s = {"x": x, "full": None}
    if case["kind"] == "pfb":
        hop, N = case["hop"], case["N"]
        s["plan"] = rfr.Plan(N, case["T"], window=case["window"], beta=case["beta"], words=words, decimation=hop,
                             full=case["full"])
        if case["full"]:
            s["full"] = torch.zeros((-(-case["n"] // hop), N), dtype=torch.complex64, device=DEV)
    elif case["kind"] == "chirp":
        hop = case["D"]
        start, rate = _chirps(case, seed)
        s["plan"] = rfr.Plan.chirp(case["L"], start, rate, window="blackman", cutoff=LOWPASS, decimation=hop)
    else:
        hop = case["D"]
        s["plan"] = rfr.Plan(0, case["L"], window="blackman", cutoff=LOWPASS, words=words, decimation=hop)
    # frames of a call: n / hop, one more now and then where n is no multiple
    s["tones"] = torch.zeros((case["tones"], -(-case["n"] // hop)), dtype=torch.complex64, device=DEV)
    return s


def prepare(case, seed):
    if case["kind"] == "tx":
        r = np.random.default_rng(seed)
        nt = case["tones"]
        words, phases = (r.integers(0, 2 ** 64 - 1, size=nt, dtype=np.uint64, endpoint=True) for _ in range(2))
        u = r.uniform(0.5, 1.0, nt)
        return {"kind": "tx", "tx": rfr.Tx(words, u * 30000.0 / u.sum(), phases), "n": case["n"], "m0": 0,
                "out": torch.zeros((case["n"], 2), dtype=torch.int16, device=DEV)}
    if case["kind"] == "batch":
        parts = [_make(c, seed * 64 + i) for i, c in enumerate(_streams(case))]
        return {"kind": "batch", "batch": rfr.Batch([p["plan"] for p in parts]), "xs": [p["x"] for p in parts],
                "fulls": [p["full"] for p in parts], "tones": [p["tones"] for p in parts]}
    return dict(_make(case, seed), kind=case["kind"])


# -------------------------------------------------------------------- run
def run(state):
    if state["kind"] == "tx":
        state["tx"].synthesize(state["m0"], state["out"])
        state["m0"] += state["n"]
        return state["out"]
    if state["kind"] == "batch":
        state["batch"].push(state["xs"], state["fulls"], state["tones"])
        return {"full": state["fulls"], "tones": state["tones"]}
    state["plan"].push_into(state["x"], state["full"], state["tones"])
    return {"full": state["full"], "tones": state["tones"]}


# ------------------------------------------------------------------- work
def work(case):
    """Input read once, outputs written once, the plan's tables read once; the FIR, the transform or the contraction."""
    if case["kind"] == "batch":
        w = [work(c) for c in _streams(case)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    n, nt = case["n"], case["tones"]
    if case["kind"] == "tx":        # a sine, a cosine and two multiply-adds for each tone and sample
        return {"bytes": 4.0 * n, "flops": 8.0 * n * nt}
    if case["kind"] == "pfb":
        N, T = case["N"], case["T"]
        F = n / case["hop"]
        return {"bytes": 4.0 * n + 8.0 * F * nt + (8.0 * F * N if case["full"] else 0.0) + 4.0 * N * T,
                "flops": F * N * (4.0 * T + 5.0 * math.log2(N))}
    F = n / case["D"]
    tables = 8.0 * case["L"] * nt if case["kind"] == "demod" else 4.0 * case["L"]
    return {"bytes": 4.0 * n + 8.0 * F * nt + tables, "flops": 8.0 * F * case["L"] * nt}


# ------------------------------------------------------------------ exact
def _lowpass(window, beta, cutoff, m):
    j = np.arange(m)
    if window == "kaiser":
        w = np.kaiser(m, beta)
    else:
        a = {"hann": (0.5, 0.5, 0.0), "hamming": (0.54, 0.46, 0.0), "blackman": (0.42, 0.5, 0.08)}[window]
        t = 2 * np.pi * j / (m - 1)
        w = a[0] - a[1] * np.cos(t) + a[2] * np.cos(2 * t)
    h = w * np.sinc(2 * cutoff * (j - (m - 1) / 2))
    return torch.from_numpy(h / h.sum()).to(DEV)


def _samples(x, lo, hi):
    """Samples lo .. hi-1 of the stream in 64 bits (0 before sample 0)."""
    z = torch.zeros(hi - lo, dtype=torch.complex128, device=DEV)
    v = x[max(lo, 0):hi].to(torch.float64)
    z[max(0, -lo):] = torch.complex(v[:, 0], v[:, 1])
    return z


def _exact_pfb(case, seed):
    words, x = _signal(case, seed)
    N, T, H, n = case["N"], case["T"], case["hop"], case["n"]
    h = _lowpass(case["window"], case["beta"], 0.5 / N, N * T).view(T, N)
    bins = torch.tensor([((int(w) * N + (1 << 63)) >> 64) % N for w in words], device=DEV)
    F = n // H
    full = torch.zeros((-(-n // H), N), dtype=torch.complex128, device=DEV) if case["full"] else None
    tones = torch.zeros((case["tones"], -(-n // H)), dtype=torch.complex128, device=DEV)
    step = max(1, (1 << 24) // N)
    for k in range(0, F, step):
        m = min(step, F - k)
        b0 = (k + 1) * H - N * T                        # first sample of frame k
        z = _samples(x, b0, b0 + (m - 1) * H + N * T)
        v = torch.zeros((m, N), dtype=torch.complex128, device=DEV)
        for t in range(T):
            v += h[t] * z.as_strided((m, N), (H, 1), t * N)
        y = torch.fft.fft(v)
        if H != N:                                      # the channel phase of the frame's absolute start
            turn = (b0 + H * torch.arange(m, device=DEV))[:, None] * torch.arange(N, device=DEV)[None, :] % N
            a = turn.to(torch.float64) * (-2 * math.pi / N)
            y *= torch.complex(torch.cos(a), torch.sin(a))
        if full is not None:
            full[k:k + m] = y
        tones[:, k:k + m] = y[:, bins].T
    return {"full": full, "tones": tones}


def _exact_demod(case, seed):
    words, x = _signal(case, seed)
    L, D, n = case["L"], case["D"], case["n"]
    h = _lowpass("blackman", 0.0, LOWPASS, L)
    F = n // D
    out = torch.zeros((case["tones"], -(-n // D)), dtype=torch.complex128, device=DEV)
    if case["kind"] == "chirp":
        start, rate = _chirps(case, seed)
        z = _samples(x, D - L, n)                       # D - L: first sample of frame 0
        m = torch.arange(D - L, n, device=DEV)
        for c in range(case["tones"]):
            s, r = (torch.tensor(int(v[c:c + 1].view(np.int64)[0]), device=DEV) for v in (start, rate))
            y = z * _turns(s * m + r * m * m).conj()
            v = torch.view_as_real(y)
            out[c, :F] = torch.complex(*(v[:, i].as_strided((F, L), (2 * D, 2), i) @ h for i in (0, 1)))
        return {"full": None, "tones": out}
    w = torch.from_numpy(words.view(np.int64)).to(DEV)
    taps = h[:, None] * _turns(torch.arange(L, device=DEV)[:, None] * w[None, :]).conj()
    step = 8192
    for k in range(0, F, step):
        m = min(step, F - k)
        b0 = (k + 1) * D - L
        z = _samples(x, b0, b0 + (m - 1) * D + L)
        y = z.as_strided((m, L), (D, 1)).contiguous() @ taps
        b = b0 + D * torch.arange(m, device=DEV)
        out[:, k:k + m] = (y * _turns(b[:, None] * w[None, :]).conj()).T
    return {"full": None, "tones": out}


def exact(case, seed):
    if case["kind"] == "tx":       # whole numbers
        return None
    if case["kind"] == "batch":
        parts = [(_exact_pfb if c["kind"] == "pfb" else _exact_demod)(c, seed * 64 + i)
                 for i, c in enumerate(_streams(case))]
        return {k: [p[k] for p in parts] for k in ("full", "tones")}
    return (_exact_pfb if case["kind"] == "pfb" else _exact_demod)(case, seed)
