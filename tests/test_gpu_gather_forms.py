"""GPU: a frustum gather's result is each pixel's own.  The same bits, the same samples and the same counts come
out of a whole frame and of a crop of it, of one frame a launch (four threads a pixel) and of enough frames for
one thread a pixel, whatever the hulls of the neighbouring pixels: long hulls along x and along y, short ones,
super-resolution, inpainting of few and of most of a frame's pixels.
"""
import dataclasses

import numpy as np
import pytest

import synth
from _gpu import Session, run_frustum, run_superres

pytestmark = pytest.mark.gpu
W, H, F, O, T = 317, 171, 61, 26, 26


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


@pytest.fixture(scope="module")
def clips():
    c = synth.make_clip("room", W, H, F, seed=12)
    c.depth[::7, 40:100, 60:140] = 0.0
    K = c.K[:, [1, 0, 2]][:, :, [1, 0, 2]]
    t = dataclasses.replace(c, W=H, H=W, K=np.ascontiguousarray(K), w2c=np.ascontiguousarray(c.w2c[:, [1, 0, 2]]),
                            rgb=np.ascontiguousarray(c.rgb.transpose(0, 2, 1, 3)),
                            depth=np.ascontiguousarray(c.depth.transpose(0, 2, 1)))
    return {"x": c, "y": t}


def _launch(sess, cid, f0, f1, crop=None, **kw):
    """Outputs of frames f0..f1-1 (of the crop) and the launch's counts, without debug records."""
    t, ss = sess.torch, sess.ss
    w, h, _ = sess.clips[cid]
    x0, y0, cw, ch = crop or (0, 0, w, h)
    p = sess.params(frame_begin=f0, frame_end=f1, crop_x=x0, crop_y=y0, crop_w=cw, crop_h=ch, gather=ss.SSVP_GATHER_FRUSTUM, **kw)
    ss.ssvp_gather_filter(sess.ctx, p, [cid])
    o = t.empty((f1 - f0, h, w, 3), dtype=t.float32, device=sess.dev)
    ss.ssvp_read_output(sess.ctx, cid, f0, f1, o)
    ss.ssvp_sync(sess.ctx)
    return o[:, y0:y0 + ch, x0:x0 + cw].cpu().numpy(), ss.ssvp_read_stats(sess.ctx)


@pytest.mark.parametrize("axis,colour_fmt,l,half_window", [("x", 0, 3.0, T), ("y", 1, 3.0, T), ("x", 1, 9.0, T), ("y", 0, 0.7, T), ("x", 0, 3.0, 4), ("x", 0, 3.0, 0)])
def test_one_frame_many_frames_and_a_crop(sess, clips, axis, colour_fmt, l, half_window):
    clip = clips[axis]
    sess.load(0, clip, colour_fmt=colour_fmt)
    kw = dict(half_window=half_window, frustum_l=l)
    # one launch of all frames takes one thread a pixel (more than one and a half waves of three CTAs an SM)
    ctas = (clip.W + 31) // 32 * ((clip.H + 7) // 8)
    n = 8
    sms = sess.torch.cuda.get_device_properties(0).multi_processor_count
    assert 2 * ctas < 3 * 3 * sms < 2 * ctas * n
    many, st = _launch(sess, 0, O, O + n, **kw)
    counts = np.zeros(2, np.int64)
    for i in range(n):
        one, s = _launch(sess, 0, O + i, O + i + 1, **kw)
        np.testing.assert_array_equal(one[0], many[i])
        counts += s[:2]
    assert counts.tolist() == list(st[:2]) and st[1] > 0
    x0, y0, cw, ch = crop = (clip.W // 3 + 1, clip.H // 4 + 3, 61, 43)
    part, _ = _launch(sess, 0, O, O + 1, crop=crop, **kw)
    np.testing.assert_array_equal(part[0], many[0, y0:y0 + ch, x0:x0 + cw])
    g = run_frustum(sess, 0, O, crop=crop, membership=True, **kw)
    np.testing.assert_array_equal(g.rgb, part[0])


@pytest.mark.parametrize("scale", [2, 3])
def test_superres_crop(sess, clips, scale):
    clip = clips["x"]
    sess.load(0, clip)
    ss = sess.ss
    whole = run_superres(sess, 0, O, scale, half_window=T)
    ew, aw, _ = ss.ssvp_read_stats(sess.ctx)
    # the same pixels in crops of other alignment: bands of rows
    cuts = [0, 37, 38, 171, clip.H * scale]
    e = a = 0
    for y0, y1 in zip(cuts[:-1], cuts[1:]):
        part = run_superres(sess, 0, O, scale, crop=(0, y0, clip.W * scale, y1 - y0), half_window=T)
        np.testing.assert_array_equal(part.rgb, whole.rgb[y0:y1])
        s = ss.ssvp_read_stats(sess.ctx)
        e, a = e + s[0], a + s[1]
    assert (e, a) == (ew, aw) and aw > 0


@pytest.mark.parametrize("mode", ["SSVP_MODE_INPAINT", "SSVP_MODE_SEMI"])
@pytest.mark.parametrize("half_window", [0, 2, 9])
@pytest.mark.parametrize("share", [0.0, 0.03, 0.9])
def test_masked_pixels(sess, mode, half_window, share):
    """Frames of few and of many masked pixels (one and four threads a pixel), bands of them, and with records."""
    clip = synth.make_clip("room", 800, 450, 25, seed=3)
    sess.load(0, clip)
    t, ss = sess.torch, sess.ss
    rng = np.random.default_rng(5)
    mask = np.zeros((25, 450, 800), np.uint8)
    mask[:, :int(450 * share), 3:] = rng.random((25, int(450 * share), 797)) < 0.97
    ss.ssvp_set_mask(sess.ctx, 0, t.from_numpy(mask).to(sess.dev))
    kw = dict(half_window=half_window, mode=getattr(ss, mode))
    whole, st = _launch(sess, 0, 12, 13, **kw)
    e = a = 0
    for y0, y1 in ((0, 37), (37, 38), (38, 150), (150, 450)):
        part, s = _launch(sess, 0, 12, 13, crop=(0, y0, 800, y1 - y0), **kw)
        np.testing.assert_array_equal(part[0], whole[0, y0:y1])
        e, a = e + s[0], a + s[1]
    assert (e, a) == st[:2]
    if share == 0.0:
        np.testing.assert_array_equal(whole[0], clip.rgb[12])
    crop = (11, 5, 64, 21)
    g = run_frustum(sess, 0, 12, crop=crop, membership=True, **kw)
    np.testing.assert_array_equal(g.rgb, whole[0, 5:26, 11:75])
