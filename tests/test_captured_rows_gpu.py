"""N = 16384 with up to 4 taps: a push captured into a caller's graph needs no
plan scratch, so the graph stays valid when a larger push outside the capture
makes the plan grow its FIR rows.  Its frames equal direct pushes' bit for bit."""
import numpy as np
import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("T,full", [(4, True), (2, False)])
def test_graph_outlives_the_rows(lib, tmp_path, T, full):
    N, nt = 16384, 21
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    F = (3 if full else 8) * sms                                 # the sums ahead, outside a capture
    rng = np.random.default_rng(T)
    x = torch.randint(-8192, 8192, (2 * F * N, 2), dtype=torch.int16, device=DEV)
    words = siggen.bin_words(rng.integers(0, N, nt), N)
    plan = lambda: lib.Plan(N, T, window="hamming", words=words, full=full)
    out = lambda n: (torch.zeros((n, N), dtype=torch.complex64, device=DEV) if full else None,
                     torch.zeros((nt, n), dtype=torch.complex64, device=DEV))
    want, got = out(F), out(F)
    ref, p = plan(), plan()
    for q in (ref, p):
        q.push_into(x[:F * N], *out(F))
    ref.push_into(x[F * N:], *want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g):
        p.push_into(x[F * N:], *got)
    g.debug_dump(str(tmp_path / "graph.dot"))
    text = (tmp_path / "graph.dot").read_text()
    assert "pfb_rows_kernel" in text and "fir_pre_kernel" not in text
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert a is None or torch.equal(a, b)
    # the plan goes on with twice the frames; the graph's frames that end inside its own
    # buffer (from T - 1 on) come out the same again
    p.push_into(x, *out(2 * F))
    for a in got:
        if a is not None:
            a.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[1][:, T - 1:], want[1][:, T - 1:])
    assert not full or torch.equal(got[0][T - 1:], want[0][T - 1:])
