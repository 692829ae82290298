"""The small-N filter banks (Sec. III.A; N = 64 .. 2048, 1 .. 16 taps) at the
edges of their tiles of 4096 / N frames: pushes of one to a few hundred frames,
split anywhere (carries of any length, buffers at any 4-byte offset), spectrum
rows of odd pitch, tones only.  One push and any split agree bit for bit, tone
rows equal their spectrum columns, and both match the FP64 oracle."""
import numpy as np
import pytest

import oracle
import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("N", [64, 128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("T,frames,first,off,pad", [
    (1, 1, 5, 0, 0), (3, 2, 64, 1, 1), (4, 65, 333, 2, 0), (7, 63, 1000, 3, 3), (8, 129, 4097, 1, 0),
    (9, 17, 7, 0, 1), (12, 64, 2049, 2, 2), (16, 200, 12345, 3, 0),
])
def test_tiles_any_split_and_oracle(lib, N, T, frames, first, off, pad):
    rng = np.random.default_rng(N + T + frames)
    n = frames * N + N // 2
    xn = rng.integers(-8192, 8192, size=(n, 2)).astype(np.int16)
    words = siggen.bin_words(rng.integers(0, N, 13), N)
    mk = lambda full: lib.Plan(N, T, window="hamming", words=words, full=full)
    buf = torch.zeros((n + off, 2), dtype=torch.int16, device=DEV)
    buf[off:] = torch.from_numpy(xn).to(DEV)
    x = buf[off:]
    ref = torch.zeros((frames, N), dtype=torch.complex64, device=DEV)
    p = mk(True)
    x0 = torch.from_numpy(xn).to(DEV)
    rt = torch.zeros((13, frames), dtype=torch.complex64, device=DEV)
    assert p.push_into(x0, ref, rt) == frames
    full = torch.zeros((frames + 1, N + pad), dtype=torch.complex64, device=DEV)
    tones = torch.zeros((13, frames + pad), dtype=torch.complex64, device=DEV)
    q = mk(True)
    cut = min(first, n)
    f0 = q.push_into(x[:cut], full, tones)
    assert f0 + (q.push_into(x[cut:], full, tones, frame_offset=f0) if cut < n else 0) == frames
    only = torch.zeros((13, frames), dtype=torch.complex64, device=DEV)
    assert mk(False).push_into(x, tones=only) == frames
    torch.cuda.synchronize()
    assert torch.equal(full[:frames, :N], ref) and torch.equal(tones[:, :frames], rt) and torch.equal(only, rt)
    assert not full[frames].any() and not full[:, N:].any() and not tones[:, frames:].any()
    assert torch.equal(rt, ref[:, torch.from_numpy(p.bins().astype(np.int64)).to(DEV)].T)
    h64, _ = oracle.pfb_prototype(N, T, "hamming")
    y = oracle.pfb(xn, N, T, h64)["full"]
    # FP32 rounding of taps, FIR and up to three passes: a few 1e-7
    assert np.linalg.norm(ref.cpu().numpy() - y) <= 1e-6 * np.linalg.norm(y)
