"""GPU: the forms of the virtual-aperture gather that a call without debug records takes (four threads a pixel in
small launches, one in large ones) against the form with records, which is compared with the oracle: the same
bits and the same counts, for window starts of every residue modulo 4 and heights that are no multiple of 2 or 8.
"""
import numpy as np
import pytest

import oracle
import synth
from _gpu import Session, compare_aperture

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


@pytest.mark.parametrize("colour_fmt", [0, 1])
@pytest.mark.parametrize("O,T,crop", [(5, 5, (3, 5, 41, 29)), (6, 5, (0, 0, 77, 45)), (7, 5, (40, 31, 33, 3)), (8, 5, (64, 8, 13, 1)),
                                      (2, 1, (5, 4, 32, 8)), (9, 0, (5, 4, 40, 15)), (10, 9, (30, 20, 20, 17))])
def test_without_records(sess, colour_fmt, O, T, crop):
    clip = synth.make_clip("planes3", 77, 45, 20, seed=5)
    if colour_fmt == 1:
        clip.rgb[:] = clip.rgb.astype(np.float16)  # what the library stores
    sess.load(0, clip, colour_fmt=colour_fmt)
    kw = dict(mode=1, k=7, half_window=T, aperture=0.08, focal_depth=0.0, cap=31, lens_samples=16)
    g = sess.run(0, O, crop=crop, membership=True, **kw)
    counts = sess.ss.ssvp_read_stats(sess.ctx)[:2]
    med = oracle.median_depth(clip.depth)
    prm = oracle.Params(mode=oracle.MODE_APERTURE, k=7, T=T, aperture=0.08, focal_depth=med, lens_samples=16, cap=31)
    s = compare_aperture(g, oracle.gather_filter(oracle.ClipView.of(clip), prm, O, crop=crop, membership=True), 31)
    assert s["members"] > 0
    plain = sess.run(0, O, crop=crop, **kw)
    np.testing.assert_array_equal(plain.rgb, g.rgb)
    assert sess.ss.ssvp_read_stats(sess.ctx)[:2] == counts


@pytest.mark.parametrize("colour_fmt", [0, 1])
@pytest.mark.parametrize("T", [0, 1, 4])
def test_many_frames_in_one_launch(sess, colour_fmt, T):
    t, ss = sess.torch, sess.ss
    W, H, n = 321, 179, 10
    clip = synth.make_clip("room", W, H, n + 2 * T, seed=2)
    sess.load(0, clip, colour_fmt=colour_fmt)
    # all frames in one launch are more than three waves of four CTAs an SM, one frame is less than one
    ctas = (W + 31) // 32 * ((H + 7) // 8)
    sms = t.cuda.get_device_properties(0).multi_processor_count
    assert ctas < 3 * sms and ctas * n > 3 * 4 * sms

    def launch(f0, f1):
        p = sess.params(mode=1, half_window=T, frame_begin=f0, frame_end=f1, aperture=0.05, cap=31, lens_samples=16)
        ss.ssvp_gather_filter(sess.ctx, p, [0])
        o = t.empty((f1 - f0, H, W, 3), dtype=t.float32, device=sess.dev)
        ss.ssvp_read_output(sess.ctx, 0, f0, f1, o)
        ss.ssvp_sync(sess.ctx)
        return o.cpu().numpy(), ss.ssvp_read_stats(sess.ctx)

    many, st = launch(T, T + n)
    counts = np.zeros(2, np.int64)
    for i in range(n):
        one, s = launch(T + i, T + i + 1)
        np.testing.assert_array_equal(one[0], many[i])
        counts += s[:2]
    assert counts.tolist() == list(st[:2]) and st[1] > 0
