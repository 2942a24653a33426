"""Wide nodes with empty child slots: their inverted boxes let no ray in, at any width."""
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


# from one leaf in the root (all other slots empty) to a few nodes whose last slots are; the first
# call comes before any refit by the caller, the second after one
@pytest.mark.parametrize("n", [2, 3, 4, 5, 7, 8])
def test_empty_slots_are_never_entered(n):
    sc = I.slab_scene(16, n=n)
    S = lt.Scene(sc)
    paths = 20011
    for lift in (None, 0.1):
        if lift is not None:
            S.refit(torch.tensor(sc.heights, dtype=torch.float32, device="cuda") + lift)
        out = []
        for width in (2, 4, 8):
            h = torch.full((paths,), 0x7FFFFFFF, dtype=torch.int32, device="cuda")
            dbg = torch.full((paths, 4), -1.0, device="cuda")
            S.primal(S.opts(seed=9, n_paths=paths, max_depth=8, hash_out=h, dbg_out=dbg, bvh_width=width))
            out.append((h, dbg))
        S.sync_status()
        for h, dbg in out[1:]:
            assert torch.equal(h, out[0][0]) and torch.equal(dbg, out[0][1])
