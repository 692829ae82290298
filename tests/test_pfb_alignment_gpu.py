"""The N = 4096 filter banks of 8 and 4 taps (Sec. III.A) on pushes of any alignment and
length: buffers that start 0 .. 3 samples into a 16-byte line, carries of any
length (the block across the carry's end), frame counts around one frame per
CTA and whole tone groups, spectrum rows of odd pitch, up to 1280 tones held on
chip and more.  Frames equal, bit for bit, one aligned push of the whole
stream, and the hop N/2 and N/4 plans (phase passes of the same kernel) too;
the aligned push matches the FP64 oracle."""
import numpy as np
import pytest

import oracle
import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
N = 4096


def _words(nt, seed):
    bins = siggen.rng_for(seed).integers(0, N, nt)
    return siggen.bin_words(bins, N)


def _stream(n, seed, off):
    """n samples starting `off` samples into a 16-byte line."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randint(-8192, 8192, (n, 2), dtype=torch.int16, generator=g)
    buf = torch.zeros((n + off, 2), dtype=torch.int16, device=DEV)
    buf[off:] = x.to(DEV)
    return buf[off:]


def _out(F, nt, pad):
    full = torch.zeros((F, N + pad), dtype=torch.complex64, device=DEV)
    return full, torch.zeros((nt, F + pad), dtype=torch.complex64, device=DEV)


@pytest.mark.parametrize("T,hop", [(8, 4096), (4, 4096), (8, 2048), (8, 1024)])
@pytest.mark.parametrize("off,first,frames,nt,pad", [
    (0, 4096, 1, 5, 0), (1, 1, 3, 1000, 0), (2, 4095, 151, 37, 1), (3, 4097, 152, 1280, 0), (1, 5000, 153, 1281, 0),
    (0, 8190, 610, 1025, 2), (3, 40000, 700, 1000, 0), (2, 3, 2500, 64, 3),
])
def test_any_alignment_equals_aligned_push(lib, T, hop, off, first, frames, nt, pad):
    n = frames * hop + 17
    words = _words(nt, 90 + nt)
    mk = lambda: lib.Plan(N, T, window="kaiser", beta=9.0, words=words, decimation=hop)
    x0 = _stream(n, 7, 0)
    ref_full, ref_tones = _out(frames, nt, 0)
    assert mk().push_into(x0, ref_full, ref_tones) == frames
    x = _stream(n, 7, off)
    p = mk()
    full, tones = _out(frames, nt, pad)
    done = 0
    for a, b in ((0, min(first, n)), (min(first, n), n)):
        if b > a:
            done += p.push_into(x[a:b], full, tones, frame_offset=done)
    torch.cuda.synchronize()
    assert done == frames
    assert torch.equal(full[:, :N], ref_full) and torch.equal(tones[:, :frames], ref_tones)
    assert not full[:, N:].any() and not tones[:, frames:].any()
    # tones only, the same stream
    q = lib.Plan(N, T, window="kaiser", beta=9.0, words=words, decimation=hop, full=False)
    t2 = torch.zeros((nt, frames), dtype=torch.complex64, device=DEV)
    assert q.push_into(x, tones=t2) == frames
    torch.cuda.synchronize()
    assert torch.equal(t2, ref_tones)
    assert torch.equal(ref_tones, ref_full[:, torch.from_numpy(p.bins().astype(np.int64)).to(DEV)].T)
    if hop == N and frames <= 200:
        h64, _ = oracle.pfb_prototype(N, T, "kaiser", 9.0)
        y = oracle.pfb(x0.cpu().numpy(), N, T, h64)["full"]
        # FP32 rounding of taps, FIR and three radix-16 passes: a few 1e-7
        got = ref_full.cpu().numpy()
        assert np.linalg.norm(got - y) <= 1e-6 * np.linalg.norm(y)
