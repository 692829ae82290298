"""Chirp demodulation with overlapping frames: segments of 128 frames a CTA and
more (hop 256), where a work item's 32 frames at most are a quarter of a segment or
less, on both sides of 128 and of the widest segment; one and two frames a CTA,
where items of one frame or the single-frame kernel are picked; filters that end
inside a block.  The check is the one of the other segments (frames against the
same frames computed one by one, bit for bit, and against the FP64 oracle)."""
import pytest

import test_chirp_overlap_gpu as overlap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,D,nc,per_cta,more", [
    (512, 256, 1, 128, 0), (512, 256, 3, 128, 1), (1024, 256, 2, 129, 0), (512, 256, 5, 191, 0), (2048, 256, 1, 185, 1),
    (1000, 256, 2, 190, 1), (512, 256, 4, 263, 7), (1920, 256, 16, 2, -4), (1920, 256, 16, 1, 0), (1920, 256, 3, 2, 0),
    (2048, 256, 7, 3, 1), (307, 256, 5, 16, 9), (3000, 1024, 9, 4, 2), (9216, 2048, 16, 1, -50),
    (15360, 2048, 2, 2, 0), (4096, 512, 2, 5, 0),
])
def test_segments(lib, L, D, nc, per_cta, more):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    overlap.test_overlapping_frames_equal_single_frames_and_oracle(lib, L, D, nc, per_cta * sms + more)
