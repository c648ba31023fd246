"""GPU: the frustum gather's long hulls, whose blocks are dropped by the depth ranges of 8 x 8 pixel tiles,
against the oracle's scan of all pixels: hulls along x and along y (the clip transposed), sizes that are
no multiple of a tile, tiles without a valid depth, hulls of a few and of many pixels across; and one
thread a pixel against four.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from _gpu import Session, compare_frustum, run_frustum

pytestmark = pytest.mark.gpu
W, H, F, O, T = 317, 171, 61, 30, 30


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
    c.depth[::7, 40:100, 60:140] = 0.0  # whole tiles without a depth in every seventh frame
    # x and y exchanged: the same geometry seen through a mirror, with hulls along y
    K = c.K[:, [1, 0, 2]][:, :, [1, 0, 2]]
    t = dataclasses.replace(c, W=H, H=W, K=np.ascontiguousarray(K), w2c=np.ascontiguousarray(c.w2c[:, [1, 0, 2]]),
                            rgb=np.ascontiguousarray(c.rgb.transpose(0, 2, 1, 3)),
                            depth=np.ascontiguousarray(c.depth.transpose(0, 2, 1)))
    return {"x": c, "y": t}


@pytest.mark.parametrize("axis", ["x", "y"])
@pytest.mark.parametrize("l,x0,y0", [(3.0, 0, 0), (3.0, 150, 80), (0.7, 309, 163), (17.0, 40, 60)])
def test_long_hulls_against_the_oracle(sess, clips, axis, l, x0, y0):
    clip = clips[axis]
    sess.load(0, clip)
    crop = (x0, y0, 8, 8) if axis == "x" else (y0, x0, 8, 8)
    prm = oracle.default_params(clip.depth, T=T)
    prm.frustum_l = l
    g = run_frustum(sess, 0, O, crop=crop, membership=True, half_window=T, frustum_l=l)
    o = oracle.frustum_filter(oracle.ClipView.of(clip), prm, O, crop=crop, membership=True)
    d = clip.depth[O, crop[1]:crop[1] + 8, crop[0]:crop[0] + 8]
    s = compare_frustum(g, o, np.isfinite(d) & (d > 0))
    assert s["members"] > 0
    if (l, x0) == (3.0, 150):  # inside the image the hulls are long: more than 32 positions of 3 pixels a frame
        assert g.nexam.max() > (2 * T + 1) * 32 * 3 // 2


def test_one_and_four_threads_a_pixel(sess, clips):
    clip = clips["x"]
    sess.load(0, clip)
    t, ss = sess.torch, sess.ss
    out = []
    for n in (1, 4):  # 220 CTAs of 32 x 8 pixels a frame: four frames in one launch take one thread a pixel
        p = sess.params(half_window=T, frame_begin=O, frame_end=O + n, gather=ss.SSVP_GATHER_FRUSTUM)
        ss.ssvp_gather_filter(sess.ctx, p, [0])
        o = t.empty((1, H, W, 3), dtype=t.float32, device=sess.dev)
        ss.ssvp_read_output(sess.ctx, 0, O, O + 1, o)
        ss.ssvp_sync(sess.ctx)
        out.append((o.cpu().numpy(), ss.ssvp_read_stats(sess.ctx)))
    # sums of up to 2^10 FP32 terms below 1 in another order
    np.testing.assert_allclose(out[0][0], out[1][0], rtol=0, atol=2.0 ** -14)
