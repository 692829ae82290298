"""N = 16384 with up to 4 taps on a full device (allocations failed by the host-side
injection): a push whose FIR rows find no room runs without them, with the same bits.
The failure is remembered, so the next push of that size does not try again; rows that
are there still serve the pushes that fit; a reset tries again."""
import numpy as np
import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def test_refused_rows_are_not_tried_again(lib):
    N, T, nt = 16384, 4, 9
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small, big = 3 * sms, 4 * sms                               # frames; both take the sums ahead
    x = torch.randint(-8192, 8192, (big * N, 2), dtype=torch.int16, device=DEV)
    words = siggen.bin_words(np.random.default_rng(1).integers(0, N, nt), N)

    def run(p, f):
        full = torch.zeros((f, N), dtype=torch.complex64, device=DEV)
        tones = torch.zeros((nt, f), dtype=torch.complex64, device=DEV)
        assert p.push_into(x[:f * N], full, tones) == f
        torch.cuda.synchronize()
        return full, tones

    sizes = [big, small, big, small, big]
    ref, p = (lib.Plan(N, T, window="hamming", words=words) for _ in range(2))
    want = [run(ref, f) for f in sizes]
    assert p.inject_alloc_failures(5) == 0
    got = [run(p, sizes[0])]
    assert p.inject_alloc_failures(0) == 4                       # tried once
    got.append(run(p, sizes[1]))                                 # fits: rows of its size
    assert p.inject_alloc_failures(5) == 0
    got += [run(p, f) for f in sizes[2:]]
    assert p.inject_alloc_failures(0) == 5                       # not tried: refused before, or there
    for a, b in zip(got, want):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    p.reset()
    assert p.inject_alloc_failures(1) == 0
    run(p, big)
    assert p.inject_alloc_failures(0) == 0                       # tried again


def test_rows_that_a_shape_needs_fail_the_push(lib):
    N, nt = 8192, 5
    words = siggen.bin_words(np.arange(nt), N)
    p = lib.Plan(N, 4, window="hamming", words=words)
    x = torch.randint(-8192, 8192, (40 * N, 2), dtype=torch.int16, device=DEV)
    full = torch.zeros((40, N), dtype=torch.complex64, device=DEV)
    tones = torch.zeros((nt, 40), dtype=torch.complex64, device=DEV)
    p.inject_alloc_failures(1)
    with pytest.raises(lib.RfrError):
        p.push_into(x, full, tones)
    assert p.info()["samples_consumed"] == 0
    assert p.push_into(x, full, tones) == 40
