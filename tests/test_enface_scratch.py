"""The scratch size of the en-face projection, on the host: sizes that the
projection refuses need none, so nothing is allocated before the refusal."""
import pytest


@pytest.mark.parametrize("w,h,d,fast_axis,taken", [
    (300, 300, 512, 0, True), (1, 1, 1, 1, True), (4096, 2, 3, 0, True), (4097, 2, 3, 0, False),
    (4097, 2, 3, 1, True), (2, 4096, 3, 1, True), (2, 4097, 3, 1, False), (2, 65535, 1, 0, True),
    (2, 65536, 1, 0, False), (65535 * 8, 2, 1, 1, True), (65535 * 8 + 1, 2, 1, 1, False), (0, 2, 3, 0, False),
    (2, 3, 4, 2, False), (2, 3, 4, -1, False)])
def test_scratch_of_accepted_and_refused_sizes(w, h, d, fast_axis, taken):
    from paper_2010_06931_gb300 import _native as N
    n = N.lib().octmc_enface_workspace(w, h, d, fast_axis)
    if taken:
        assert n >= 2 * 4 * w * h * d  # two volumes and the small buffers
        assert n <= 2 * 4 * w * h * d + 16 * max(w, h) + (1 << 20)
    else:
        assert n == -1
