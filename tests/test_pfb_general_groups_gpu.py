"""Two-pass filter banks (N = N1 N2) whose CTAs take several groups in a row, the next
group's points on their way while a group's last stage runs: one, two, three and four
stages a pass, rows of even and odd length, both CTA sizes; spectrum only, tones only
and both.  The three agree bit for bit, and frames match the definition in FP64."""
import numpy as np
import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("N,T,frames", [
    (8748, 2, 500), (10000, 4, 400), (16807, 3, 300), (20000, 4, 300), (33614, 2, 150), (65536, 2, 120), (78125, 4, 60),
    (90000, 3, 60), (131072, 4, 40), (250000, 2, 30), (1000000, 1, 9), (1500000, 2, 6),
])
def test_groups_in_a_row(lib, N, T, frames):
    rng = np.random.default_rng(N)
    x = torch.randint(-8192, 8192, (frames * N + 5, 2), dtype=torch.int16, device=DEV)
    words = siggen.bin_words(rng.permutation(N)[:700], N)
    plan = lambda **k: lib.Plan(N, T, window="hamming", words=words, **k)
    full = lambda: torch.zeros((frames, N), dtype=torch.complex64, device=DEV)
    tones = lambda: torch.zeros((len(words), frames), dtype=torch.complex64, device=DEV)
    both, only_full, only_tones = (full(), tones()), full(), tones()
    p = plan()
    assert p.push_into(x, *both) == frames
    assert plan(tones=False).push_into(x, full=only_full) == frames
    assert plan(full=False).push_into(x, tones=only_tones) == frames
    torch.cuda.synchronize()
    bins = torch.from_numpy(p.bins().astype(np.int64)).to(DEV)
    assert torch.equal(only_full, both[0]) and torch.equal(only_tones, both[1])
    assert torch.equal(both[1], both[0][:, bins].T)
    h = torch.from_numpy(p.taps_table()[1].astype(np.float64)).to(DEV).view(T, N)
    z = torch.view_as_complex(x.to(torch.float64))
    for k in sorted({0, T, frames // 2, frames - 1}):
        v = torch.zeros(N, dtype=torch.complex128, device=DEV)
        for t in range(T):
            lo = (k + 1 - T + t) * N
            if lo >= 0:
                v += h[t] * z[lo:lo + N]
        ref = torch.fft.fft(v)
        assert (both[0][k] - ref).norm() <= 1e-6 * ref.norm()
