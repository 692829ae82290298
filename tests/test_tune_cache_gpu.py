"""Launch choices of another product form, or of a cache file written before the
three-product GEMM's form was picked by size, never pin a plan's form."""
import json
import re

import pytest

import siggen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
L, D, NT, FRAMES = 4096, 256, 256, 94 * 128


def _plan(lib):
    words = siggen.demod_case(1 << 12, NT, seed=5)["words"]
    return lib.Plan(0, L, window="blackman", cutoff=1e-3, words=words, decimation=D)


def _kernels(plan, tmp_path):
    """The GEMM kernels a push launches: those of a captured push's graph."""
    x = torch.zeros((FRAMES * D, 2), dtype=torch.int16, device=DEV)
    out = torch.zeros((NT, FRAMES), dtype=torch.complex64, device=DEV)
    plan.push_into(x, tones=out)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g):
        plan.push_into(x, tones=out)
    path = tmp_path / "graph.dot"
    g.debug_dump(str(path))
    text = path.read_text()
    return set(re.findall(r"demod3m_gemm_kernelI\w+?EE|combine3_kernel", text))


def test_choice_of_the_other_form_pins_nothing(lib, tmp_path, monkeypatch):
    monkeypatch.setenv("RFR_TUNE_CACHE", str(tmp_path / "tune.json"))
    by_size = _kernels(_plan(lib), tmp_path)
    # by size this push takes pairs, which a pinned tone tile excludes
    pinned = _plan(lib)
    pinned.set_tone_tile(128)
    assert by_size and _kernels(pinned, tmp_path) != by_size
    p = _plan(lib)
    p.set_demod_products(4)
    assert p.autotune(FRAMES * D) > 0
    p.set_demod_products(3)
    assert _kernels(p, tmp_path) == by_size
    # and the other form's entry is not this one's
    assert p.autotune(FRAMES * D) > 0
    assert len(json.loads((tmp_path / "tune.json").read_text())) == 2


def test_entries_of_the_older_format_are_not_found(lib, tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("RFR_TUNE_CACHE", str(path))
    prop = torch.cuda.get_device_properties(0)
    lg = (FRAMES * D).bit_length() - 1
    old = f"demod:N0:T0:L{L}:D{D}:tones{NT}:flags2:n2^{lg}:sm{prop.major}{prop.minor}x{prop.multi_processor_count}"
    path.write_text('{\n  "%s": [0, 19, 64, 0, 0, 0]\n}\n' % old)
    p = _plan(lib)
    assert p.autotune(FRAMES * D) > 0                        # timed, not loaded
    q = _plan(lib)
    assert q.autotune(FRAMES * D) == -1.0
    assert q.tune() == p.tune()
    assert old in json.loads(path.read_text())               # an older program still finds its own


def test_look_ahead_is_timed_for_the_ring_kernel_only(lib, tmp_path, monkeypatch):
    monkeypatch.setenv("RFR_TUNE_CACHE", str(tmp_path / "tune.json"))
    for N, T, hop, ring in ((256, 8, 256, False), (4096, 8, 4096, False), (4096, 8, 1024, False), (8192, 16, 8192, False),
                            (1000, 4, 1000, False), (32, 8, 32, True), (2048, 4, 2048, True), (4096, 6, 4096, True)):
        p = lib.Plan(N, T, window="hamming", words=siggen.bin_words([1, 2], N), decimation=hop)
        assert p.autotune(1 << 16) > 0
        assert p.tune()["pfb_lookahead"] in ((1, 2, 3) if ring else (0,))
        q = lib.Plan(N, T, window="hamming", words=siggen.bin_words([1, 2], N), decimation=hop)
        assert q.autotune(1 << 16) == -1.0 and q.tune() == p.tune()
