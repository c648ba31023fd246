"""GPU: a training gradient depends on the samples of its sets alone, not on what an earlier call left in the
unused slots: the gradient of a batch whose sets are short, computed after one call that filled every slot
with finite colours and after one that filled them with infinite ones, is the same.  Both ways of
extracting the sets: by a list (two pixels of many) and with the whole frame (half of a small frame's pixels).
"""
import numpy as np
import pytest

import oracle
import synth
from _gpu import Session

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


@pytest.mark.parametrize("W,H,n", [(64, 40, 2), (16, 10, 80)])
def test_unused_slots_do_not_reach_the_gradient(sess, W, H, n):
    t, ss = sess.torch, sess.ss
    clip = synth.make_clip("planes3", W, H, 5, seed=3)
    O, T, k = 2, 2, 5
    sess.load(0, clip)
    sess.load(1, clip, rgb=np.full_like(clip.rgb, np.inf))
    ss.ssvp_set_mlp(sess.ctx, *oracle.he_init(2))
    clean = t.from_numpy(clip.clean).to(sess.dev)
    p = sess.params(k=k, half_window=T, frame_begin=O, frame_end=O + 1, radius=-0.005)
    wide = sess.params(k=k, half_window=T, frame_begin=O, frame_end=O + 1, radius=-0.5)
    counts = []
    for prm in (p, wide):
        feat, col = t.zeros((W * H, 64, 16), dtype=t.int16, device=sess.dev), t.zeros((W * H, 64, 3), device=sess.dev)
        ns, plain = t.zeros(W * H, dtype=t.int32, device=sess.dev), t.zeros((W * H, 3), device=sess.dev)
        ss.ssvp_learned_samples(sess.ctx, prm, 0, feat, col, ns, plain)
        ss.ssvp_sync(sess.ctx)
        counts.append(ns.cpu().numpy())
    short = np.flatnonzero((counts[0] > 0) & (counts[0] < 50) & (counts[1] == 64))
    # one pixel repeated: every CTA's share of the sums is the same, so their order does not matter
    idx = np.full(n, short[len(short) // 2], np.int32)

    def grad(cid, prm):
        return ss.ssvp_mlp_grad(sess.ctx, prm, cid, idx, clean)

    grad(0, wide)
    want = grad(0, p)
    grad(1, wide)
    got = grad(0, p)
    assert np.isfinite(want).all() and np.abs(want[:1216]).max() > 0
    assert np.isfinite(got).all(), got[1218]
    # W1, b1, W2 and the loss to the bit; b2's two sums join four warps' parts in any order
    np.testing.assert_array_equal(got[:1216], want[:1216])
    assert got[1218] == want[1218]
    np.testing.assert_allclose(got[1216:1218], want[1216:1218], rtol=1e-3, atol=1e-6)
