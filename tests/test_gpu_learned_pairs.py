"""GPU: the learned filter's sample sets of a crop large enough to be stored in pairs, against those of a crop
of the same rows small enough to be stored one by one: the same counts, features, colours and plain result,
to the bit (both crops start at the same pixel, so their tiles and geometry are the same).
"""
import numpy as np
import pytest

import synth
from _gpu import Session

pytestmark = pytest.mark.gpu
W, H, ROWS = 640, 480, 464  # 307,200 pixels and 296,960


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


@pytest.mark.parametrize("k,T,colour_fmt", [(1, 0, 0), (3, 2, 1), (5, 1, 0), (7, 3, 0), (7, 2, 1)])
def test_pairs_and_single_stores_agree(sess, k, T, colour_fmt):
    t = sess.torch
    clip = synth.make_clip("room", W, H, 2 * T + 1, seed=6)
    clip.depth[T, 100:140, 200:300] = 0.0  # pixels without a set
    sess.load(0, clip, colour_fmt=colour_fmt)

    def sets(rows):
        n = W * rows
        feat = t.zeros((n, 64, 16), dtype=t.int16, device=sess.dev)
        col = t.zeros((n, 64, 3), dtype=t.float32, device=sess.dev)
        ns = t.zeros(n, dtype=t.int32, device=sess.dev)
        plain = t.zeros((n, 3), dtype=t.float32, device=sess.dev)
        p = sess.params(k=k, half_window=T, frame_begin=T, frame_end=T + 1, crop_x=0, crop_y=0, crop_w=W, crop_h=rows)
        sess.ss.ssvp_learned_samples(sess.ctx, p, 0, feat, col, ns, plain)
        sess.ss.ssvp_sync(sess.ctx)
        return feat, col, ns, plain

    one, two = sets(ROWS), sets(H)
    n = W * ROWS
    held = t.arange(64, device=sess.dev)[None] < one[2][:, None]
    assert t.equal(one[2], two[2][:n]) and t.equal(one[3], two[3][:n])
    assert t.equal(one[0][held], two[0][:n][held]) and t.equal(one[1][held], two[1][:n][held])
    counts = set(np.unique(one[2].cpu().numpy()) & 1)
    assert counts == {0, 1}  # sets that end on either half of a pair
