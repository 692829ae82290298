"""N = 16384 with up to 4 taps: a push captured into a caller's graph stays valid when
a larger push outside the capture makes the plan grow its FIR rows: the rows that
the graph uses stay as long as the plan.  Its frames equal direct pushes' bit for bit,
and memory allocated after the growth is left alone by its replays."""
import numpy as np
import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("T,full", [(4, True), (2, False)])
def test_graph_outlives_the_rows(lib, T, full):
    N, nt = 16384, 21
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    F = (3 if full else 8) * sms                                 # the sums ahead
    rng = np.random.default_rng(T)
    x = torch.randint(-8192, 8192, (2 * F * N, 2), dtype=torch.int16, device=DEV)
    words = siggen.bin_words(rng.integers(0, N, nt), N)
    plan = lambda: lib.Plan(N, T, window="hamming", words=words, full=full)
    out = lambda n: (torch.zeros((n, N), dtype=torch.complex64, device=DEV) if full else None,
                     torch.zeros((nt, n), dtype=torch.complex64, device=DEV))
    want, got, later = out(F), out(F), out(2 * F)
    ref, p = plan(), plan()
    for q in (ref, p):
        q.push_into(x[:F * N], *out(F))
    ref.push_into(x[F * N:], *want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.push_into(x[F * N:], *got)
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert a is None or torch.equal(a, b)
    # the plan grows twice; then the graph's frames that end inside its own buffer (from
    # T - 1 on) come out the same again
    p.push_into(x[:(F + 1) * N], *later)
    p.push_into(x, *later)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    guard = torch.full((min(free // 2, 4 * F * N * 8),), 0x5a, dtype=torch.uint8, device=DEV)
    for a in got:
        if a is not None:
            a.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[1][:, T - 1:], want[1][:, T - 1:])
    assert not full or torch.equal(got[0][T - 1:], want[0][T - 1:])
    assert (guard == 0x5a).all()
