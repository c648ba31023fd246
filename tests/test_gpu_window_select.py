"""GPU: the window gather's test loop, which drops candidates before the exact radius test, keeps every
sample: membership against the oracle for radii from a fraction of a pixel to more than the window (the
depth-only and the whole-distance test and the line between them), window starts of both parities, ragged
sizes, windows across the image's edges; and the kernel without debug outputs gives the same colours.
"""
import numpy as np
import pytest

import oracle
import synth
from _gpu import Session, compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sess():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    s = Session()
    yield s
    s.close()


@pytest.mark.parametrize("k", [1, 3, 5, 7, 9])
@pytest.mark.parametrize("r_px", [0.4, 1.7, 2.5, 9.0])
def test_survivors_hold_every_sample(sess, k, r_px):
    clip = synth.make_clip("room", 71, 43, 5, seed=9)  # odd sizes: windows start at odd and even columns
    sess.load(0, clip)
    median = oracle.median_depth(clip.depth)
    radius = np.float32(r_px * median / clip.K[0, 0, 0])  # r_px pixels at the median depth
    view = oracle.ClipView.of(clip)
    prm = oracle.Params(mode=oracle.MODE_DENOISE, k=k, T=2, radius=float(radius))
    members = 0
    for O in (0, 2):
        g = sess.run(0, O, membership=True, k=k, half_window=2, radius=float(radius))
        o = oracle.gather_filter(view, prm, O, membership=True)
        members += compare(g, o, k)["members"]
        # the same template without the records: at most 5 * 81 FP32 terms of size < 1 a sum
        plain = sess.run(0, O, k=k, half_window=2, radius=float(radius))
        np.testing.assert_allclose(plain.rgb, g.rgb, rtol=0, atol=405 * 2.0 ** -24)
    assert members >= 2 * 71 * 43  # at least the pixels themselves


@pytest.mark.parametrize("T", [30, 40, 50, 60, 127])
def test_staged_long_windows(sess, T):
    """Windows whose geometry and staged boxes come near, to and over 48 KB of shared memory."""
    clip = synth.make_clip("planes3", 45, 37, 9, seed=2)
    sess.load(0, clip)
    a = sess.run(0, 4, k=5, half_window=T)
    b = sess.run(0, 4, k=5, half_window=T, gather=sess.ss.SSVP_GATHER_WINDOW_TMA)
    np.testing.assert_array_equal(a.rgb, b.rgb)
