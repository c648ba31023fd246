"""GPU: gradients of small batches, whose sample sets are extracted by a pixel list (one warp a pixel),
element by element against the oracle: k from 1 to 7, windows of one frame to more frames than a warp has
lanes, both colour formats, a batch of one pixel, the frame's last pixel, a pixel without a valid depth.
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
@pytest.mark.parametrize("k,T,n", [(1, 0, 1), (3, 2, 37), (5, 8, 301), (7, 17, 200)])
def test_gradients_of_a_pixel_list(sess, colour_fmt, k, T, n):
    clip = synth.make_clip("planes3", 71, 43, 37, seed=4)  # T = 17: 35 window frames, two rounds of 32 lanes
    O = 18
    if colour_fmt == 1:
        clip.rgb[:] = clip.rgb.astype(np.float16)  # what the library stores
    clip.depth[O, 20, 30] = 0.0
    sess.load(0, clip, colour_fmt=colour_fmt)
    prm = oracle.default_params(clip.depth, k=k, T=T, radius_rel=0.02)
    W1, b1, W2, _ = oracle.he_init(6)
    b2 = np.array([0.1, 0.0])
    sess.ss.ssvp_set_mlp(sess.ctx, W1, b1, W2, b2)
    of, oc, on, op = oracle.learned_crop(oracle.ClipView.of(clip), prm, O)
    flags = _flags(clip, prm, O, (0, 0, clip.W, clip.H))
    clean = clip.clean[O].astype(np.float64)
    # pixels without a membership ambiguity and with a clear BCE target (as in the whole-frame test)
    cand = []
    for y in range(clip.H):
        for x in range(clip.W):
            if flags[y, x] or on[y, x] < 1:
                continue
            ol, _, _, _ = oracle.mlp_pixel(of[y, x], oc[y, x], on[y, x], W1, b1, W2, b2, plain=op[y, x])
            el, ep = np.mean((ol - clean[y, x]) ** 2), np.mean((op[y, x] - clean[y, x]) ** 2)
            # with one sample both outputs are that sample: the target is 1 up to rounding
            if abs(el - ep) > 1e-3 * max(el, ep, 1e-12):
                cand.append((y, x))
    if k == 1 and T == 0:
        cand = [(20, 30)]  # the pixel without a depth: no set, no gradient
    rng = np.random.default_rng(n)
    pick = [cand[i] for i in rng.choice(len(cand), size=n, replace=len(cand) < n)]
    if n > 1:
        pick[-1] = (20, 30)
    idx = np.array([y * clip.W + x for y, x in pick], np.int32)
    assert 4 * n < clip.W * clip.H  # few enough to go by the list
    p = sess.params(k=k, half_window=T, frame_begin=O, frame_end=O + 1, radius=-0.02)
    g = sess.ss.ssvp_mlp_grad(sess.ctx, p, 0, idx, sess.torch.from_numpy(clip.clean).to(sess.dev))
    ys, xs = zip(*pick)
    L, gW1, gb1, gW2, gb2, aW1, ab1, aW2, ab2 = oracle.mlp_loss_grad(
        of[ys, xs], oc[ys, xs], on[ys, xs], op[ys, xs], clean[ys, xs], W1, b1, W2, b2, round_bf16=True, term_scale=True)
    assert g[1218] == pytest.approx(L, rel=1e-4, abs=1e-12)
    # the bound of the whole-frame test: 1e-3 |oracle| + c (sum of |terms| of the entry) + 1e-6 (largest such sum), c
    # covering FP32 accumulation and, for the tensor-core products, their BF16 operands (2^-8 of each term)
    bf = 2.0 ** -8 + 2e-4
    for got, want, scale, c in ((g[:1024], gW1.ravel(), aW1.ravel(), bf), (g[1024:1088], gb1, ab1, bf),
                                (g[1088:1216], gW2.ravel(), aW2.ravel(), bf), (g[1216:1218], gb2, ab2, 2e-4)):
        err = np.abs(got - want)
        tol = 1e-3 * np.abs(want) + c * scale + 1e-6 * scale.max()
        assert (err <= tol).all(), (np.flatnonzero(err > tol)[:5], err.max(), tol.max())
