"""GPU: the frustum gather's instances that drop whole blocks of long hulls, which windows and images of some size
take, against the oracle's scan of all pixels: hulls along x and along y (the clip transposed), two band widths,
super-resolution, inpainting and semi-transparency; and the same bits with one thread a pixel and with four.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from _gpu import Session, compare_frustum, run_frustum, run_superres, superres_ref_valid

pytestmark = pytest.mark.gpu
W, H, F, O, T = 832, 96, 68, 30, 30


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
    c.depth[::7, 20:60, 160:340] = 0.0  # whole tiles without a depth in every seventh frame
    K = c.K[:, [1, 0, 2]][:, :, [1, 0, 2]]
    t = dataclasses.replace(c, W=H, H=W, K=np.ascontiguousarray(K), w2c=np.ascontiguousarray(c.w2c[:, [1, 0, 2]]),
                            rgb=np.ascontiguousarray(c.rgb.transpose(0, 2, 1, 3)),
                            depth=np.ascontiguousarray(c.depth.transpose(0, 2, 1)))
    return {"x": c, "y": t}


def _turn(axis, x0, y0, n=8):
    return (x0, y0, n, n) if axis == "x" else (y0, x0, n, n)


def _hull_length(clip, J):
    """Length in pixels that the ray of frame O's centre projects to in frame J, over J's depth range: 32 and more are
    walked by blocks."""
    d = clip.depth[J]
    d = d[np.isfinite(d) & (d > 0)]
    z = np.geomspace(0.01, 1000.0, 20001)
    x = np.linalg.inv(clip.K[O]) @ np.array([clip.W / 2, clip.H / 2, 1.0])
    w = clip.w2c.reshape(clip.F, -1, 4)[:, :3]
    X = w[O, :, :3].T @ (x[:, None] * z - w[O, :, 3:])
    q = clip.K[J] @ (w[J, :, :3] @ X + w[J, :, 3:])
    q = q[:, (q[2] >= d.min()) & (q[2] <= d.max())]
    return float(np.abs(q[:2] / q[2] - (q[:2] / q[2])[:, :1]).max()) if q.shape[1] else 0.0


@pytest.mark.parametrize("axis,l,x0,y0", [("x", 3.0, 400, 40), ("y", 3.0, 400, 40), ("x", 3.0, 0, 0), ("y", 9.0, 823, 87), ("x", 9.0, 300, 20)])
def test_against_the_oracle(sess, clips, axis, l, x0, y0):
    clip, crop = clips[axis], _turn(axis, x0, y0)
    sess.load(0, clip)
    prm = oracle.default_params(clip.depth, T=T)
    prm.frustum_l = l
    g = run_frustum(sess, 0, O, crop=crop, membership=True, half_window=T, frustum_l=l)
    o = oracle.frustum_filter(oracle.ClipView.of(clip), prm, O, crop=crop, membership=True)
    d = clip.depth[O, crop[1]:crop[1] + 8, crop[0]:crop[0] + 8]
    s = compare_frustum(g, o, np.isfinite(d) & (d > 0))
    assert s["members"] > 0
    assert sum(_hull_length(clip, J) > 33 for J in range(O - T, O + T + 1)) > 10


@pytest.mark.parametrize("axis,colour_fmt,l", [("x", 0, 3.0), ("y", 1, 3.0), ("x", 1, 9.0)])
def test_one_and_four_threads_a_pixel(sess, clips, axis, colour_fmt, l):
    t, ss = sess.torch, sess.ss
    clip = clips[axis]
    sess.load(0, clip, colour_fmt=colour_fmt)
    ctas, n = (clip.W + 31) // 32 * ((clip.H + 7) // 8), 8
    sms = t.cuda.get_device_properties(0).multi_processor_count
    assert 2 * ctas < 3 * 3 * sms < 2 * ctas * n

    def launch(f0, f1):
        p = sess.params(half_window=T, frame_begin=f0, frame_end=f1, gather=ss.SSVP_GATHER_FRUSTUM, frustum_l=l)
        ss.ssvp_gather_filter(sess.ctx, p, [0])
        o = t.empty((f1 - f0, clip.H, clip.W, 3), dtype=t.float32, device=sess.dev)
        ss.ssvp_read_output(sess.ctx, 0, f0, f1, o)
        ss.ssvp_sync(sess.ctx)
        return o.cpu().numpy(), ss.ssvp_read_stats(sess.ctx)

    many, st = launch(O, O + n)
    counts = np.zeros(2, np.int64)
    for i in range(n):
        one, s = launch(O + i, O + i + 1)
        np.testing.assert_array_equal(one[0], many[i])
        counts += s[:2]
    assert counts.tolist() == list(st[:2]) and st[1] > 0
    x0, y0, cw, ch = crop = _turn(axis, 411, 33, 30)
    g = run_frustum(sess, 0, O, crop=crop, membership=True, half_window=T, frustum_l=l)
    np.testing.assert_array_equal(g.rgb, many[0, y0:y0 + ch, x0:x0 + cw])


def test_superres(sess, clips):
    clip = clips["x"]
    sess.load(0, clip)
    med = oracle.median_depth(clip.depth)
    p = oracle.Params(mode=0, k=1, T=T, radius=0.005 * med, sigma_rgb=50.0 / 255.0, sigma_xyz=0.03 * med,
                      gather=oracle.GATHER_FRUSTUM, frustum_l=6.0)
    crop = (801, 77, 8, 8)
    g = run_superres(sess, 0, O, 2, crop=crop, membership=True, half_window=T, mode=0, frustum_l=6.0, sigma_rgb=p.sigma_rgb,
                     sigma_xyz=p.sigma_xyz)
    o = oracle.superres_filter(oracle.ClipView.of(clip), p, O, 2, crop=crop, membership=True)
    assert compare_frustum(g, o, superres_ref_valid(clip, O, 2, crop))["members"] > 0


@pytest.mark.parametrize("semi", [False, True])
def test_masked_pixels(sess, clips, semi):
    clip, crop = clips["x"], _turn("x", 400, 40)
    sess.load(1, clip)
    rng = np.random.default_rng(3)
    mask = (rng.random((F, H, W)) < 0.7).astype(np.uint8)
    sess.ss.ssvp_set_mask(sess.ctx, 1, mask)
    masked = mask[O, 40:48, 400:408] != 0
    sigma_rgb, sigma_xyz = (80.0 / 255.0, 0.03 * oracle.median_depth(clip.depth)) if semi else (55.0 / 255.0, 0.0)
    prm = oracle.Params(mode=oracle.MODE_DENOISE, k=1, T=T, radius=0.01, sigma_rgb=sigma_rgb, sigma_xyz=sigma_xyz,
                        gather=oracle.GATHER_FRUSTUM, frustum_l=3.0)
    g = run_frustum(sess, 1, O, crop=crop, membership=True, half_window=T, sigma_rgb=sigma_rgb, sigma_xyz=sigma_xyz,
                    mode=sess.ss.SSVP_MODE_SEMI if semi else sess.ss.SSVP_MODE_INPAINT)
    o = oracle.inpaint_filter(oracle.ClipView.of(clip), prm, mask, O, crop=crop, membership=True, semi=semi)
    s = compare_frustum(g, o, masked)
    assert s["members"] > 0
    np.testing.assert_array_equal(g.rgb[~masked], clip.rgb[O, 40:48, 400:408][~masked])
