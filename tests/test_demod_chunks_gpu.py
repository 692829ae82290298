"""The accumulation chunk of the three-product form: every setting is its own
rounding, and a shorter chunk is closer to the FP64 oracle (the tensor cores'
internal accumulation error grows with the sums that a chunk collects)."""
import numpy as np
import pytest

import oracle
import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("nt,L,D,frames", [(24, 1024, 512, 400), (300, 960, 64, 3000)])
def test_shorter_chunks_are_closer(lib, nt, L, D, frames):
    c = siggen.demod_case(frames * D, nt, seed=77 + nt)
    x = torch.from_numpy(c["x"]).to(DEV)
    some = np.linspace(0, nt - 1, 24).astype(int)
    ref = oracle.demod(c["x"], L, D, oracle.lowpass("blackman", L, 1e-3), c["words"][some])
    err, outs = [], []
    for k in (1, 2, 3, 4, 8):
        p = lib.Plan(0, L, window="blackman", cutoff=1e-3, words=c["words"], decimation=D)
        p.set_accum_chunk(k)
        out = torch.zeros((nt, frames), dtype=torch.complex64, device=DEV)
        assert p.push_into(x, tones=out) == frames
        torch.cuda.synchronize()
        outs.append(out)
        err.append(np.linalg.norm(out[some].cpu().numpy() - ref) / np.linalg.norm(ref))
    for a, b in zip(outs, outs[1:]):
        assert not torch.equal(a, b)
    assert all(a < b for a, b in zip(err, err[1:])), err
    # the default is 4
    p = lib.Plan(0, L, window="blackman", cutoff=1e-3, words=c["words"], decimation=D)
    out = torch.zeros((nt, frames), dtype=torch.complex64, device=DEV)
    p.push_into(x, tones=out)
    torch.cuda.synchronize()
    assert torch.equal(out, outs[3])
