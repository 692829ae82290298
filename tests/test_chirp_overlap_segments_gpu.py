"""Chirp demodulation with overlapping frames, hop 256: segments of 128 frames
a CTA and more, where a work item's 32 frames at most are a quarter of a
segment or less; frame counts a CTA on both sides of 128 and of the widest
segment.  The check is the one of the shorter segments (frames against the
same frames computed one by one, bit for bit, and against the FP64 oracle)."""
import pytest

import test_chirp_overlap_gpu as overlap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nc,per_cta,more", [
    (512, 1, 128, 0), (512, 3, 128, 1), (1024, 2, 129, 0), (512, 5, 191, 0), (2048, 1, 185, 1),
    (1000, 2, 190, 1), (512, 4, 263, 7),
])
def test_long_segments(lib, L, nc, per_cta, more):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    overlap.test_overlapping_frames_equal_single_frames_and_oracle(lib, L, 256, nc, per_cta * sms + more)
