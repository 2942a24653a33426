"""A backward call leaves what the primal recorded as it is: several calls after one primal, with
other image adjoints, scatter modes and with or without the recorded masks, give the gradients of
the fused form, which keeps nothing between calls; so do batched passes and the autotuner's runs.
Paths whose last connection lies beyond the hits that a record holds, and paths with one."""
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


def adjoint(S, seed):
    return torch.tensor(I.smooth_adjoint(S.W, S.H, seed), dtype=torch.float32, device="cuda")


def close(got, ref):
    # FP32 sums of the same per-path terms in another order: 1e-5 as in the other replays' tests
    for a, b in zip(got, ref):
        assert rel_l2(a, b) < 1e-5


# at most 32 vertices have one word of validity bits, and more recorded hits
@pytest.mark.parametrize("scene,depth,n", [("box_3bit", 64, 4099), ("box_3bit", 32, 4099), ("box_7bit", 40, 8191),
                                           ("slab_in_box_11bit", 33, 8191), ("slab_in_box_11bit", 32, 8191),
                                           ("slab_17bit", 12, 40001)])
@pytest.mark.parametrize("attached", [0, 1])
def test_calls_after_one_primal(scene, depth, n, attached):
    S = lt.Scene(SCENES[scene]())
    kw = dict(seed=9, n_paths=n, max_depth=depth, attached=attached)
    state = S.new_lrb3_state(n)
    S.primal(S.opts(lrb3_state=state, **kw))
    rows = []
    # adjoint, scatter mode, masks known
    for k, scatter, ready in [(1, 0, 1), (2, 0, 1), (3, 2, 1), (2, 0, 0), (1, 0, 1)]:
        dI = adjoint(S, k)
        dbg = torch.zeros((n, 4), device="cuda")
        got = S.backward_lrb3(S.opts(lrb3_state=state, lrb3_mask_ready=ready, scatter=scatter, dbg_out=dbg, **kw), dI)
        close(got, S.backward_lrb3(S.opts(**kw), dI))
        rows.append(dbg)
    S.sync_status()
    # delta_total and the number of connections of each path: the same arithmetic at each call
    assert torch.equal(rows[0], rows[4]) and torch.equal(rows[1], rows[3])
    assert (rows[0][:, 3] > 1).any() and (rows[0][:, 3] == 1).any()


@pytest.mark.parametrize("scene,depth,n", [("box_3bit", 64, 4099), ("box_7bit", 12, 20011), ("slab_17bit", 12, 40001)])
@pytest.mark.parametrize("attached", [0, 1])
def test_buffered_calls_after_one_primal(scene, depth, n, attached):
    S = lt.Scene(SCENES[scene]())
    kw = dict(seed=9, n_paths=n, max_depth=depth, attached=attached)
    o = S.opts(**kw)
    buf = torch.empty(S.lrb2_buffer_bytes(o), dtype=torch.uint8, device="cuda")
    S.primal(o, estimator=lt.EST_BUFFERED, aux=buf)
    for k, scatter in [(1, 0), (2, 0), (3, 2), (1, 0)]:
        dI = adjoint(S, k)
        close(S.backward_lrb2(S.opts(scatter=scatter, **kw), dI, buf), S.backward_lrb3(o, dI))
    S.sync_status()


def batch_items(**kw):
    specs = [(I.box_scene(32), dict(n_paths=3000, max_depth=40, seed=1)),
             (I.box_scene(48, heightmap=8, hm_std=0.03), dict(n_paths=5001, max_depth=40, seed=2, attached=1)),
             (I.slab_scene(64, n=12, seed=2), dict(n_paths=20011, max_depth=6, seed=3, attached=1))]
    items = []
    for k, (sc, o) in enumerate(specs):
        S = lt.Scene(sc)
        items.append(dict(scene=S, d_image=adjoint(S, 100 + k), **o, **kw))
    return items


def check_batch(items):
    torch.cuda.synchronize()
    for it in items:
        S = it["scene"]
        o = S.opts(seed=it["seed"], n_paths=it["n_paths"], max_depth=it["max_depth"], attached=it.get("attached", 0))
        close(it["grads"], S.backward_lrb3(o, it["d_image"]))
        S.sync_status()


def test_batched_pass_after_one_primal():
    B = lt.Batch(batch_items(lrb3_state=True))
    B.run(lt.PASS_PRIMAL)
    for seed in (1, 2, 3):
        for k, it in enumerate(B.items):
            it["d_image"].copy_(adjoint(it["scene"], 100 * seed + k))
        B.run(lt.PASS_LRB3)
        check_batch(B.items)


def test_batch_reads_a_state_of_a_batch_without_known_masks(monkeypatch):
    """The primal pass records the same whatever the batch's own LRB-3 pass would use: here it is
    run by a batch with an item that has no state, and read by one whose items all have."""
    items = batch_items(lrb3_state=True)
    B = lt.Batch(items + [dict(items[0], lrb3_state=False)])
    B.run(lt.PASS_PRIMAL)
    states = [it["_state"] for it in items]
    second = batch_items(lrb3_state=True)
    given = iter(states)
    monkeypatch.setattr(lt.Scene, "new_lrb3_state", lambda self, n: next(given))
    B2 = lt.Batch(second)
    B2.run(lt.PASS_LRB3)
    check_batch(second)
    B.run(lt.PASS_LRB3)  # fused: some item has no state
    check_batch(B.items)


def test_tuned_pass_holds_one_complete_run():
    B = lt.Batch(batch_items(lrb3_state=True))
    B.run(lt.PASS_PRIMAL)
    B.tune(lt.PASS_LRB3, reps=1)
    check_batch(B.items)
