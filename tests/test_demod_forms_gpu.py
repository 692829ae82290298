"""The forms of the three-product demodulation GEMM (Sec. III.B) at the edges
of their tiles: the form picked by size (two-SM tiles, single-CTA tiles, each
product a work item of its own when tiles are few), the pinned two-SM form and
single-CTA tiles of 128 tones give the same frames bit for bit (the same MMAs
in the same order), and match the FP64 oracle within the readout's tolerance
(relative RMS error <= 1e-5 per tone)."""
import numpy as np
import pytest

import oracle
import siggen
from helpers import TOL, rel_rows

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"

# L, D, tones, frames: tone widths around the steps of 16 and 32 and the tile
# widths 128 and 256, frames around the tile heights 128 and 256, one and many
# chunks of taps, several tiles per CTA (the parked tiles' ring)
SHAPES = [
    (64, 64, 1, 1), (64, 64, 17, 127), (128, 64, 33, 128), (200, 128, 129, 129), (1024, 512, 255, 255),
    (1024, 512, 257, 256), (1000, 448, 300, 257), (1024, 2048, 511, 513), (4096, 512, 128, 385),
    (256, 64, 1500, 9001), (192, 64, 700, 20011),
]


@pytest.mark.parametrize("L,D,nt,frames", SHAPES)
def test_forms_agree_and_match_oracle(lib, L, D, nt, frames):
    n = frames * D + D // 3
    rng = np.random.default_rng(L + D + nt + frames)
    words = siggen.random_words(rng, nt)
    x = torch.from_numpy(rng.integers(-8192, 8192, size=(n, 2)).astype(np.int16)).to(DEV)
    outs = []
    for form in ("size", "pair", "single"):
        p = lib.Plan(0, L, window="hann", cutoff=1e-3, words=words, decimation=D)
        if form != "size":
            p.set_demod_pair(form == "pair")
        out = torch.full((nt, frames + 1), 7.0, dtype=torch.complex64, device=DEV)
        # two pushes: the second one's frames start at any place of the 128-frame anchors
        cut = (frames // 3) * D + 5
        f0 = p.push_into(x[:cut], tones=out)
        assert f0 + p.push_into(x[cut:], tones=out, frame_offset=f0) == frames
        torch.cuda.synchronize()
        outs.append(out.cpu().numpy())
    assert np.all(outs[0][:, frames] == 7.0)                 # nothing past the last frame
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
    sel = np.unique(np.linspace(0, nt - 1, 6).astype(int))
    k = min(frames, 300)
    ref = oracle.demod(x.cpu().numpy()[:k * D], L, D, oracle.lowpass("hann", L, 1e-3), words[sel])
    assert rel_rows(outs[0][sel, :k], ref).max() < TOL
