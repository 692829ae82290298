"""Demodulation against chirps (Sec. III.C) with overlapping frames: every
mixer value serves all the frames that use its sample.  Frame J k + J - 1 of a
plan with hop D is frame k of the same plan with hop J D >= L, whose frames do
not overlap and are computed one by one: the two agree bit for bit, at chirp
counts around the four workers, frame counts around one per SM and several
segments, filters that end inside a block, and match the FP64 oracle."""
import numpy as np
import pytest

import oracle
import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("L,D,nc,frames", [
    (512, 256, 1, 1), (511, 256, 3, 153), (257, 256, 5, 40), (1024, 512, 4, 6000), (1500, 512, 2, 31),
    (4096, 2048, 8, 320), (4096, 512, 9, 400), (16384, 4096, 2, 170), (2000, 256, 13, 65),
])
def test_overlapping_frames_equal_single_frames_and_oracle(lib, L, D, nc, frames):
    rng = np.random.default_rng(L + D + nc)
    J = -(-L // D)
    n = frames * D + 77
    xn = rng.integers(-8192, 8192, size=(n, 2)).astype(np.int16)
    x = torch.from_numpy(xn).to(DEV)
    sw = siggen.random_words(rng, nc)
    rw = rng.integers(0, 2 ** 42, nc).astype(np.uint64)
    mk = lambda hop: lib.Plan.chirp(L, sw, rw, window="hann", cutoff=1e-3, decimation=hop)
    out = torch.zeros((nc, frames), dtype=torch.complex64, device=DEV)
    p = mk(D)
    cut = min(n, (frames // 3) * D + 19)                 # two pushes, the second behind an odd carry
    f0 = p.push_into(x[:cut], tones=out)
    assert f0 + p.push_into(x[cut:], tones=out, frame_offset=f0) == frames
    one = torch.zeros((nc, max(1, frames // J)), dtype=torch.complex64, device=DEV)
    m = mk(J * D).push_into(x, tones=one)
    torch.cuda.synchronize()
    assert torch.equal(out[:, J - 1::J][:, :m], one[:, :m])
    k = min(frames, 40)
    ref = oracle.chirp_demod(xn[:k * D], L, D, oracle.lowpass("hann", L, 1e-3), sw, rw)
    got = out[:, :k].cpu().numpy()
    # FP32 mixer and sums: a few 1e-7 of the frames' norm
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


def test_mixer_error_bound(lib):
    """With one tap of weight 1 and samples (8191, 0) a frame is 8191 exp(-i p(m)):
    the mixer itself.  Bound: phase rounding pi 2^-27, the two series' rounding
    (a few half units of 2^-24) and the product's 2^-24, 2.5e-7 in all; phases
    anywhere, and within a few units of every quadrant's edges."""
    D, frames = 64, 4096
    rng = np.random.default_rng(3)
    edges = [(q << 62) + d for q in range(4) for d in (-(1 << 33), -1, 0, 1, 1 << 32)]
    edges += [(q << 62) + (1 << 61) + d for q in range(4) for d in (-(1 << 33), -1, 0, 1, 1 << 32)]
    # frame k's sample is m = (k + 1) D - 1: a start word w gives phase w m
    sw = np.array([e * pow(2 * D - 1, -1, 1 << 64) % (1 << 64) for e in edges], np.uint64)   # phase e at frame 1
    sw = np.concatenate([sw, siggen.random_words(rng, 24)])
    rw = np.concatenate([np.zeros(len(edges), np.uint64), rng.integers(0, 2 ** 50, 24).astype(np.uint64)])
    x = torch.zeros((frames * D, 2), dtype=torch.int16, device=DEV)
    x[:, 0] = 8191
    p = lib.Plan.chirp(1, sw, rw, window="rect", decimation=D)
    out = torch.zeros((len(sw), frames), dtype=torch.complex64, device=DEV)
    assert p.push_into(x, tones=out) == frames
    got = out.cpu().numpy() / 8191.0
    m = (np.arange(frames, dtype=np.uint64) + np.uint64(1)) * np.uint64(D) - np.uint64(1)
    with np.errstate(over="ignore"):
        ph = sw[:, None] * m[None, :] + rw[:, None] * (m * m)[None, :]
    ang = ph.view(np.int64).astype(np.float64) * (np.pi / 2.0 ** 63)
    assert np.abs(got - np.exp(-1j * ang)).max() <= 2.5e-7
