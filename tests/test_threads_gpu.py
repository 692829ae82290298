"""Plans of one kernel in several host threads: three plans of small pushes and
one whose launches of the same kernel need more shared memory push beside each
other, each in a thread and on a stream of its own.  Every push succeeds and
every output is what the plan gives alone."""
import sys
import threading

import numpy as np
import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _pfb(lib, N, T, nt, n):
    words = [lib.freq_to_word(k * 200e6 / N, 200e6) for k in range(nt)]
    return lib.Plan(N, T, window="kaiser", beta=9.0, words=words, full=False), n, nt, N


def _chirp(lib, L, D, n):
    w = siggen.random_words(np.random.default_rng(L + D), 2)
    return lib.Plan.chirp(L, w, w >> np.uint64(24), window="hann", cutoff=1e-3, decimation=D), n, 2, D


SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1
CASES = {
    # no tones kept on chip / 1000 of them (56 KB)
    "rows": lambda lib, big: _pfb(lib, 4096, 16, 1000, 4096 * 32 * (SMS + 1)) if big else _pfb(lib, 4096, 16, 16, 1 << 14),
    "symmetric": lambda lib, big: _pfb(lib, 4096, 8, 1500 if big else 1, 1 << 14),
    # segments of 40 frames / of one
    "chirp overlap": lambda lib, big: _chirp(lib, 1024, 512, 512 * 40 * SMS if big else 1 << 13),
    "chirp": lambda lib, big: _chirp(lib, 16384, 16384, 1 << 16) if big else _chirp(lib, 6500, 8192, 1 << 15),
    "mixed radix": lambda lib, big: _pfb(lib, 4000 if big else 100, 4, 4, 16000),
}


@pytest.mark.parametrize("case", list(CASES))
def test_threads_share_a_kernel(lib, case):
    parts = [CASES[case](lib, i == 0) for i in range(4)]
    x = torch.randint(-8192, 8192, (max(p[1] for p in parts), 2), dtype=torch.int16, device=DEV)
    want, got, errors = [], [], []
    for plan, n, nt, hop in parts:
        got.append(torch.zeros((nt, n // hop), dtype=torch.complex64, device=DEV))
        plan.push_into(x[:n], tones=got[-1])
        torch.cuda.synchronize()
        want.append(got[-1].clone())
    start, done = threading.Barrier(4), threading.Event()

    def work(i):
        plan, n, nt, hop = parts[i]
        stream = torch.cuda.Stream()
        try:
            start.wait()
            left = 12000
            while left and (i == 0 or not done.is_set()):
                plan.push_into(x[:n], tones=got[i], stream=stream)
                left -= i == 0
                if left % 256 == 255:
                    stream.synchronize()
            stream.synchronize()
            plan.reset()
            got[i].zero_()
            torch.cuda.synchronize()
            plan.push_into(x[:n], tones=got[i], stream=stream)
            stream.synchronize()
        except Exception as e:                                   # noqa: BLE001 (reported below)
            errors.append(e)
        finally:
            done.set()

    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        sys.setswitchinterval(interval)
    assert not errors
    for g, w in zip(got, want):
        assert torch.equal(g, w)
