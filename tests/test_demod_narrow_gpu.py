"""The three-product GEMM's forms at short filters and at the edges of their tiles:
tones around the 16, 32, 64, 128 and 256 wide tiles, frames around 128 and 256,
output rows of odd pitch and offset.  The form picked by size, the pinned pair, tone
tiles and fused pre-split agree bit for bit, nothing outside the frames is
written, and the frames match the FP64 oracle."""
import numpy as np
import pytest

import oracle
import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("L,D,nt,frames,fo,pad", [
    (64, 64, 1, 1, 0, 0), (64, 64, 33, 129, 1, 0), (256, 64, 16, 128, 0, 1), (256, 64, 127, 3000, 2, 0),
    (256, 64, 129, 257, 0, 0), (256, 64, 300, 20001, 1, 1), (200, 128, 64, 255, 0, 2), (1024, 512, 65, 256, 3, 0),
    (1024, 512, 96, 40000, 0, 1), (1024, 64, 257, 1500, 0, 0), (700, 64, 160, 6000, 5, 0), (2048, 512, 520, 700, 0, 1),
])
def test_forms_agree(lib, L, D, nt, frames, fo, pad):
    c = siggen.demod_case(frames * D + 11, nt, seed=L + nt)
    x = torch.from_numpy(c["x"]).to(DEV)
    cut = min(x.shape[0], (frames // 3) * D + 17)

    def run(pin):
        p = lib.Plan(0, L, window="blackman", cutoff=1e-3, words=c["words"], decimation=D)
        pin(p)
        out = torch.full((nt, fo + frames + pad), -7.0, dtype=torch.complex64, device=DEV)
        f = p.push_into(x[:cut], tones=out, frame_offset=fo)       # the rest behind an odd carry
        assert f + p.push_into(x[cut:], tones=out, frame_offset=fo + f) == frames
        torch.cuda.synchronize()
        assert (out[:, :fo] == -7).all() and (out[:, fo + frames:] == -7).all()
        return out[:, fo:fo + frames]

    want = run(lambda p: None)
    for pin in (lambda p: p.set_demod_pair(True), lambda p: p.set_tone_tile(128), lambda p: p.set_tone_tile(64),
                lambda p: p.set_fused_presplit(True)):
        assert torch.equal(run(pin), want)
    some, k = np.linspace(0, nt - 1, min(nt, 12)).astype(int), min(frames, 300)
    ref = oracle.demod(c["x"][:k * D], L, D, oracle.lowpass("blackman", L, 1e-3), c["words"][some])
    got = want[some][:, :k].cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
