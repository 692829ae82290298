"""Device memory of three-product demodulation plans: the scratch that finished
products are parked in is sized by the pushes, not for the whole chip at creation,
and a batch's one launch has its own.  Frames of small and large pushes, alone and
batched in either order, are bit-identical."""
import numpy as np
import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
L, D = 1024, 512


def _plan(lib, nt, seed):
    words = siggen.random_words(np.random.default_rng(seed), nt)
    return lib.Plan(0, L, window="blackman", cutoff=1e-3, words=words, decimation=D)


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_a_small_plan_stays_small(lib):
    n = 1 << 18
    x = torch.randint(-8192, 8192, (n, 2), dtype=torch.int16, device=DEV)
    out = torch.zeros((64, n // D), dtype=torch.complex64, device=DEV)
    _plan(lib, 64, 0).push_into(x, tones=out)                # modules loaded
    before = _used()
    plans = [_plan(lib, 64, k) for k in range(4)]
    created = _used() - before
    for p in plans:
        p.push_into(x, tones=out)
    # a plan's tables are below 1 MB, its planes of the stream 3 MB, the scratch of
    # five CTAs 2.5 MB; device memory is handed out in pages of 2 MB
    assert created <= 4 * (16 << 20)
    assert _used() - before <= 4 * (32 << 20)


@pytest.mark.parametrize("sizes", [(3, 40000, 200), (40000, 3, 129), (1000, 1000, 1000)])
@pytest.mark.parametrize("nt", [(17, 64, 300), (300, 65, 1)])
def test_batch_and_growth_equal_alone(lib, sizes, nt):
    xs = [torch.randint(-8192, 8192, (f * D + 5, 2), dtype=torch.int16, device=DEV) for f in sizes]
    out = lambda: [torch.zeros((t, f + 1), dtype=torch.complex64, device=DEV) for t, f in zip(nt, sizes)]
    alone, batched, grown = out(), out(), out()
    for k in range(3):
        _plan(lib, nt[k], k).push_into(xs[k], tones=alone[k])
    plans = [_plan(lib, nt[k], k) for k in range(3)]
    b = lib.Batch(plans)
    b.push([x[:D] for x in xs], None, batched)                   # a step of one frame each
    b.push([x[D:] for x in xs], None, batched, frame_offsets=[1, 1, 1])
    for k in range(3):                                           # pushes of 1, 2, 4, ... frames, then the rest
        p, pos, f, step = _plan(lib, nt[k], k), 0, 0, 1
        while pos < xs[k].shape[0]:
            cnt = min(step * D, xs[k].shape[0] - pos)
            f += p.push_into(xs[k][pos:pos + cnt], tones=grown[k], frame_offset=f)
            pos, step = pos + cnt, step * 2
        assert f == sizes[k]
    torch.cuda.synchronize()
    for a, c, g in zip(alone, batched, grown):
        assert torch.equal(a, c) and torch.equal(a, g)
