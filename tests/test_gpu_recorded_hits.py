"""The per-path records of the LRB-3 state and of the buffered two-pass buffer hold the
primitives of a path's first vertices: passes that intersect those give the gradients of
passes that search the scene at every vertex.  Scenes whose primitive indices take few bits
(many hits fit), many (a hit crosses a word of the record), and paths that outlast the record."""
import numpy as np
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu

SCENES = {
    "box_3bit": lambda: I.box_scene(48),
    "box_7bit": lambda: I.box_scene(48, heightmap=8, hm_std=0.03),
    "slab_in_box_11bit": lambda: I.slab_in_box(48, n=24),
    "slab_17bit": lambda: I.slab_scene(48, n=190),
}


def rel_l2(a, b):
    a, b = a.double().cpu().numpy(), b.double().cpu().numpy()
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


@pytest.mark.parametrize("scene,depth,n", [("box_3bit", 64, 4099), ("box_7bit", 40, 8191), ("slab_in_box_11bit", 33, 8191),
                                           ("slab_17bit", 12, 40001)])
@pytest.mark.parametrize("attached", [0, 1])
def test_recorded_hits_give_the_searched_gradients(scene, depth, n, attached):
    S = lt.Scene(SCENES[scene]())
    dI = torch.tensor(I.smooth_adjoint(S.W, S.H, 5), dtype=torch.float32, device="cuda")
    kw = dict(seed=9, n_paths=n, max_depth=depth, attached=attached)
    state = S.new_lrb3_state(n)
    S.primal(S.opts(lrb3_state=state, **kw))
    got = S.backward_lrb3(S.opts(lrb3_state=state, lrb3_mask_ready=1, **kw), dI)
    ref = S.backward_lrb3(S.opts(lrb3_state=S.new_lrb3_state(n), **kw), dI)  # searches in both passes
    o = S.opts(**kw)
    buf = torch.empty(S.lrb2_buffer_bytes(o), dtype=torch.uint8, device="cuda")
    S.primal(o, estimator=lt.EST_BUFFERED, aux=buf)
    got2 = S.backward_lrb2(o, dI, buf)
    S.sync_status()
    # FP32 sums of the same per-path terms in another order: 1e-5 as in the other replays' tests
    for a, b, r in zip(got, got2, ref):
        assert rel_l2(a, r) < 1e-5
        assert rel_l2(b, r) < 1e-5
