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
