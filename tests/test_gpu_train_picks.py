"""GPU: gradients of batches whose sample sets are extracted by a pixel list, element by element against the oracle, for
picks that are easily got wrong: one pixel alone, the frame's four corners, pixels with more samples than a set
holds.  The bound is that of the other gradient tests.
"""
import numpy as np
import pytest

import oracle
import synth
from _gpu import Session
from test_gpu_learned import _flags

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
@pytest.mark.parametrize("k,T,radius_rel", [(3, 2, 0.02), (7, 17, 0.05)])
def test_gradients_of_single_pixels_corners_and_full_sets(sess, colour_fmt, k, T, radius_rel):
    W, H, O = 71, 43, 18
    clip = synth.make_clip("planes3", W, H, 37, seed=4)
    if colour_fmt == 1:
        clip.rgb[:] = clip.rgb.astype(np.float16)  # what the library stores
    sess.load(0, clip, colour_fmt=colour_fmt)
    prm = oracle.default_params(clip.depth, k=k, T=T, radius_rel=radius_rel)
    W1, b1, W2, _ = oracle.he_init(6)
    b2 = np.array([0.1, 0.0])
    sess.ss.ssvp_set_mlp(sess.ctx, W1, b1, W2, b2)
    of, oc, on, op = oracle.learned_crop(oracle.ClipView.of(clip), prm, O)
    flags = _flags(clip, prm, O, (0, 0, W, H))
    clean = clip.clean[O].astype(np.float64)

    def clear(y, x):  # no membership ambiguity, a clear confidence target (as in the other gradient tests)
        if flags[y, x] or on[y, x] < 1:
            return False
        ol, _, _, _ = oracle.mlp_pixel(of[y, x], oc[y, x], on[y, x], W1, b1, W2, b2, plain=op[y, x])
        el, ep = np.mean((ol - clean[y, x]) ** 2), np.mean((op[y, x] - clean[y, x]) ** 2)
        return abs(el - ep) > 1e-3 * max(el, ep, 1e-12)

    corners = [c for c in ((0, 0), (0, W - 1), (H - 1, 0), (H - 1, W - 1)) if clear(*c)]
    full = [(y, x) for y in range(0, H, 3) for x in range(0, W, 3) if on[y, x] == 64 and clear(y, x)][:40]
    assert corners and (k == 3 or len(full) >= 8)
    batches = [[c] for c in corners] + [corners] + ([full, full[:1]] if full else [])
    p = sess.params(k=k, half_window=T, frame_begin=O, frame_end=O + 1, radius=-radius_rel)
    dev = sess.torch.from_numpy(clip.clean).to(sess.dev)
    bf = 2.0 ** -8 + 2e-4
    for pick in batches:
        idx = np.array([y * W + x for y, x in pick], np.int32)
        assert 4 * len(idx) < W * H  # few enough to go by the list
        g = sess.ss.ssvp_mlp_grad(sess.ctx, p, 0, idx, dev)
        ys, xs = zip(*pick)
        L, gW1, gb1, gW2, gb2, aW1, ab1, aW2, ab2 = oracle.mlp_loss_grad(
            of[ys, xs], oc[ys, xs], on[ys, xs], op[ys, xs], clean[ys, xs], W1, b1, W2, b2, round_bf16=True, term_scale=True)
        assert g[1218] == pytest.approx(L, rel=1e-4, abs=1e-12)
        for got, want, scale, c in ((g[:1024], gW1.ravel(), aW1.ravel(), bf), (g[1024:1088], gb1, ab1, bf),
                                    (g[1088:1216], gW2.ravel(), aW2.ravel(), bf), (g[1216:1218], gb2, ab2, 2e-4)):
            err = np.abs(got - want)
            tol = 1e-3 * np.abs(want) + c * scale + 1e-6 * scale.max()
            assert (err <= tol).all(), (pick[:2], np.flatnonzero(err > tol)[:5], err.max(), tol.max())
