"""Calls large enough for the path order (more than 512 paths per SM): the order is built, leaves out
the paths that end on their first ray, and every path has its outputs; calls at the line and below
have none.  Sizes around the blocks of its sort (1024 paths each, at most 256 blocks)."""
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


def align(x):
    return (x + 255) & ~255


def counters(state, n):
    """The five counters of the state: list length, two tickets, paths with several connections, length
    of the order."""
    at = align(32 * n) + 3 * align(4 * n)
    return state[at:at + 40].view(torch.int64).cpu().tolist()


def line():
    return 512 * torch.cuda.get_device_properties(0).multi_processor_count


SCENES = {"box": lambda: I.box_scene(32), "box_hm": lambda: I.box_scene(32, heightmap=8),
          "slab": lambda: I.slab_scene(32, n=8)}


# every BVH width (each has its own first-ray test), a scene without a BVH, and heights that move
# the BVH's box
@pytest.mark.parametrize("scene", ["box", "box_hm", "slab"])
@pytest.mark.parametrize("width", [2, 4, 8])
def test_paths_left_out_have_their_outputs(scene, width):
    sc = SCENES[scene]()
    S = lt.Scene(sc)
    n = line() + 1021
    mask = (torch.arange(n, device="cuda") % 3 != 0).to(torch.uint8)
    for lift in (0.0, 0.15):
        if S.n_heights:
            S.refit(torch.tensor(sc.heights, dtype=torch.float32, device="cuda") + lift)
        state = S.new_lrb3_state(n)
        state.fill_(0xAB)
        out = []
        for st in (None, state):
            h = torch.full((n,), 0x7FFFFFFF, dtype=torch.int32, device="cuda")
            dbg = torch.full((n, 4), -1.0, device="cuda")
            img = S.primal(S.opts(seed=5, n_paths=n, max_depth=6, lrb3_state=st, hash_out=h, dbg_out=dbg, mask=mask,
                                  bvh_width=width))
            out.append((h, dbg, img))
        S.sync_status()
        ended = int((out[0][1][:, 1] == 0).sum())  # no vertex
        length = counters(state, n)[4]
        # the order holds every path that hits something, and on the slab, where most first rays
        # leave the scene, fewer than all
        assert n - ended <= length <= n and length > 0
        if scene == "slab":
            assert ended > n // 4 and length < n
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        assert torch.allclose(out[0][2], out[1][2], rtol=1e-5, atol=1e-7)
        # validity words: a bit per valid connection of an unmasked path, zero elsewhere
        words = state[align(32 * n):align(32 * n) + 4 * n].view(torch.int32).cpu().numpy().view("uint32")
        bits = sum(((words >> k) & 1) for k in range(32))
        want = torch.where(mask > 0, out[1][1][:, 0], torch.zeros(1, device="cuda")).cpu().numpy()
        assert (bits == want).all()
        assert counters(state, n)[0] == int((want > 0).sum())


@pytest.mark.parametrize("extra", [0, 1, 1023, 1024, 1025, 33 * 1024 + 7])
def test_every_path_is_taken_once_around_the_line(extra):
    S = lt.Scene(SCENES["slab"]())
    n = line() + extra
    state = S.new_lrb3_state(n)
    sentinel = 0x7FFFFFFF
    h = torch.full((n,), sentinel, dtype=torch.int32, device="cuda")
    ref = torch.full((n,), sentinel, dtype=torch.int32, device="cuda")
    kw = dict(seed=3, path_offset=11, n_paths=n, max_depth=3)
    S.primal(S.opts(lrb3_state=state, hash_out=h, **kw))
    S.primal(S.opts(hash_out=ref, **kw))
    S.sync_status()
    assert (counters(state, n)[4] > 0) == (extra > 0)  # none at the line itself
    assert not (ref == sentinel).any()
    assert torch.equal(h, ref)


@pytest.mark.parametrize("scene", ["box_hm", "slab"])
def test_gradients_with_and_without_the_order(scene):
    """One call over the whole range (an order) against the sum of calls below the line (none)."""
    S = lt.Scene(SCENES[scene]())
    n = line() + 3001
    dI = torch.tensor(I.smooth_adjoint(S.W, S.H, 5), dtype=torch.float32, device="cuda")

    def backward(off, cnt):
        st = S.new_lrb3_state(cnt)
        kw = dict(seed=5, path_offset=off, n_paths=cnt, n_norm=n, max_depth=6, attached=1)
        S.primal(S.opts(lrb3_state=st, **kw))
        return [g.double().cpu() for g in S.backward_lrb3(S.opts(lrb3_state=st, lrb3_mask_ready=1, **kw), dI)]

    whole, a, b = backward(0, n), backward(0, n // 2), backward(n // 2, n - n // 2)
    S.sync_status()
    for w, x, y in zip(whole, a, b):
        # FP32 sums of the same per-path terms in another order: 1e-5 as in the replays' tests
        assert (w - x - y).norm() <= 1e-5 * (x + y).norm()
