"""The order in which the plain primal given the LRB-3 state takes its paths (a counting sort):
every path is taken once, at sizes around the sort's blocks."""
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


# one path; one block of the sort, its edge, two blocks; more row entries than a warp; the
# largest number of blocks, and ranges longer than one block's share
@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, 33 * 4096 + 5, 256 * 4096, 256 * 4096 + 1, (1 << 21) + 77])
def test_every_path_is_taken_once(n):
    S = lt.Scene(I.slab_scene(32, n=8))
    state = S.new_lrb3_state(n)
    # a path left out keeps the sentinel, which no decision hash of these paths equals
    sentinel = 0x7FFFFFFF
    h = torch.full((n,), sentinel, dtype=torch.int32, device="cuda")
    ref = torch.full((n,), sentinel, dtype=torch.int32, device="cuda")
    kw = dict(seed=3, path_offset=11, n_paths=n, max_depth=3)
    S.primal(S.opts(lrb3_state=state, hash_out=h, **kw))
    S.primal(S.opts(hash_out=ref, **kw))
    S.sync_status()
    assert not (ref == sentinel).any()
    assert torch.equal(h, ref)


# every BVH width (each has its own first-ray test), a scene without a BVH, and heights that move
# the BVH's box; masked paths and per-path outputs of the paths that the order leaves out
@pytest.mark.parametrize("scene", ["box", "box_hm", "slab"])
@pytest.mark.parametrize("width", [2, 4, 8])
def test_paths_left_out_of_the_order_have_their_outputs(scene, width):
    sc = {"box": lambda: I.box_scene(32), "box_hm": lambda: I.box_scene(32, heightmap=8),
          "slab": lambda: I.slab_scene(32, n=8)}[scene]()
    S = lt.Scene(sc)
    n = 50021
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
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        assert torch.allclose(out[0][2], out[1][2], rtol=1e-5, atol=1e-7)
        # validity words: a bit per valid connection of an unmasked path, zero elsewhere
        lo = 32 * n + (-32 * n) % 256
        words = state[lo:lo + 4 * n].view(torch.int32).cpu().numpy().view("uint32")
        bits = sum(((words >> k) & 1) for k in range(32))
        want = torch.where(mask > 0, out[1][1][:, 0], torch.zeros(1, device="cuda")).cpu().numpy()
        assert (bits == want).all()
