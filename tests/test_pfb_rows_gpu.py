"""The filter banks whose FIR sums go through memory (Sec. III.A; N = 4096 with
9 .. 16 taps, N = 8192 and 16384): pushes of one frame to several frames per CTA,
split anywhere, buffers at any 4-byte offset, spectrum rows that leave by TMA and
rows of odd pitch that cannot, tones only.  Every form agrees bit for bit, tone
rows equal their spectrum columns, and both match the FP64 oracle."""
import numpy as np
import pytest

import oracle
import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("N,T,frames,first,off,pad", [
    (4096, 9, 1, 4095, 0, 1), (4096, 16, 620, 100001, 1, 1), (4096, 12, 7, 3, 2, 3),
    (8192, 1, 2, 8191, 3, 1), (8192, 4, 305, 5, 1, 1), (8192, 8, 310, 700000, 0, 3), (8192, 13, 5, 9000, 2, 1),
    (16384, 3, 153, 16385, 1, 1), (16384, 4, 330, 5000000, 1, 3),
    (16384, 8, 160, 1234567, 3, 1), (16384, 16, 3, 20000, 2, 5),
])
def test_rows_any_split_pitch_and_oracle(lib, N, T, frames, first, off, pad):
    rng = np.random.default_rng(N + T + frames)
    n = frames * N + N // 3
    xn = rng.integers(-8192, 8192, size=(n, 2)).astype(np.int16)
    nt = 37
    words = siggen.bin_words(rng.integers(0, N, nt), N)
    mk = lambda full: lib.Plan(N, T, window="hamming", words=words, full=full)
    buf = torch.zeros((n + off, 2), dtype=torch.int16, device=DEV)
    buf[off:] = torch.from_numpy(xn).to(DEV)
    x = buf[off:]
    ref = torch.zeros((frames, N), dtype=torch.complex64, device=DEV)
    rt = torch.zeros((nt, frames), dtype=torch.complex64, device=DEV)
    p = mk(True)
    assert p.push_into(torch.from_numpy(xn).to(DEV), ref, rt) == frames
    full = torch.zeros((frames + 1, N + pad), dtype=torch.complex64, device=DEV)
    tones = torch.zeros((nt, frames + pad), dtype=torch.complex64, device=DEV)
    q = mk(True)
    cut = min(first, n)
    f0 = q.push_into(x[:cut], full, tones)
    assert f0 + (q.push_into(x[cut:], full, tones, frame_offset=f0) if cut < n else 0) == frames
    only = torch.zeros((nt, frames), dtype=torch.complex64, device=DEV)
    assert mk(False).push_into(x, tones=only) == frames
    torch.cuda.synchronize()
    assert torch.equal(full[:frames, :N], ref) and torch.equal(tones[:, :frames], rt) and torch.equal(only, rt)
    assert not full[frames].any() and not full[:, N:].any() and not tones[:, frames:].any()
    assert torch.equal(rt, ref[:, torch.from_numpy(p.bins().astype(np.int64)).to(DEV)].T)
    k = min(frames, 12)
    h64, _ = oracle.pfb_prototype(N, T, "hamming")
    y = oracle.pfb(xn[:k * N], N, T, h64)["full"]
    # FP32 rounding of taps, FIR and up to four passes: a few 1e-7
    assert np.linalg.norm(ref[:k].cpu().numpy() - y) <= 1e-6 * np.linalg.norm(y)


@pytest.mark.parametrize("T,frames,cut", [(1, 1, 16384), (3, 155, 16387), (4, 307, 100001)])
def test_captured_push_of_a_plan_without_rows(lib, T, frames, cut):
    """N = 16384, T <= 4: a push captured before the plan has room for its FIR sums
    (after none, or after a smaller push) runs the FIR in the FFT kernel; the replay's
    frames equal a direct push's bit for bit, and the state goes on from there."""
    N, nt = 16384, 37
    rng = np.random.default_rng(T)
    xn = rng.integers(-8192, 8192, size=(cut + frames * N, 2)).astype(np.int16)
    x = torch.from_numpy(xn).to(DEV)
    words = siggen.bin_words(rng.integers(0, N, nt), N)
    F = x.shape[0] // N
    out = lambda: (torch.zeros((F, N), dtype=torch.complex64, device=DEV),
                   torch.zeros((nt, F), dtype=torch.complex64, device=DEV))
    want, got = out(), out()
    assert lib.Plan(N, T, window="hamming", words=words).push_into(x, *want) == F
    p = lib.Plan(N, T, window="hamming", words=words)
    f0 = p.push_into(x[:cut], *got) if T > 1 else 0
    rest = x[cut:] if T > 1 else x
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert f0 + p.push_into(rest, *got, frame_offset=f0, stream=s) == F
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("N,T,frames,nt,off,pad,fo", [
    (4096, 9, 2500, 1500, 0, 0, 0), (4096, 16, 1219, 1100, 0, 2, 3), (4096, 11, 1300, 40, 1, 3, 1),
    (8192, 8, 1000, 2500, 0, 1, 2), (8192, 5, 911, 77, 1, 1, 3), (16384, 8, 470, 4300, 0, 2, 1), (16384, 4, 457, 5, 1, 2, 0),
])
def test_rows_tones_in_groups(lib, N, T, frames, nt, off, pad, fo):
    """Tone rows written four frames at a time: ranges that begin and end inside a
    group, more tones than the kernel keeps on chip, any frame offset, row pitch and
    8-byte offset of the rows.  Every value equals its spectrum bin; nothing else is
    written."""
    rng = np.random.default_rng(nt)
    x = torch.from_numpy(rng.integers(-8192, 8192, size=(frames * N, 2)).astype(np.int16)).to(DEV)
    words = siggen.bin_words(rng.integers(0, N, nt), N)
    p = lib.Plan(N, T, window="hamming", words=words)
    full = torch.zeros((fo + frames, N), dtype=torch.complex64, device=DEV)
    ld = fo + frames + pad
    base = torch.zeros(nt * ld + off, dtype=torch.complex64, device=DEV)
    tones = base[off:].view(nt, ld)
    assert p.push_into(x, full, tones, frame_offset=fo) == frames
    torch.cuda.synchronize()
    bins = torch.from_numpy(p.bins().astype(np.int64)).to(DEV)
    assert torch.equal(tones[:, fo:fo + frames], full[fo:, bins].T)
    assert not tones[:, :fo].any() and not tones[:, fo + frames:].any() and not base[:off].any()
