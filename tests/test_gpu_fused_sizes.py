"""The fused LRB-3 form without chains replays along known hits in calls of at most 128 paths per SM
and searches again in larger ones: both sides of that line against the separate-pass form."""
import numpy as np
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("attached", [0, 1])
@pytest.mark.parametrize("width", [2, 4, 8])
def test_fused_form_on_both_sides_of_a_small_call(attached, width):
    S = lt.Scene(I.box_scene(48, heightmap=8, hm_std=0.03))
    dI = torch.tensor(I.smooth_adjoint(S.W, S.H, 5), dtype=torch.float32, device="cuda")
    line = 128 * torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, 33, line, line + 1):
        kw = dict(seed=9, n_paths=n, max_depth=12, attached=attached, bvh_width=width)
        got = S.backward_lrb3(S.opts(**kw), dI)
        ref = S.backward_lrb3(S.opts(lrb3_state=S.new_lrb3_state(n), **kw), dI)
        for a, b in zip(got, ref):
            a, b = a.double().cpu().numpy(), b.double().cpu().numpy()
            # FP32 sums of the same per-path terms in another order: 1e-5 as in the replays' tests
            assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
    S.sync_status()
