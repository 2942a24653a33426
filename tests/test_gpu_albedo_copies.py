"""The albedo gradient of LRB-3 pass 3 spread over copies: textures of one texel, of sizes that
are no power of two, and too large for copies to fit, against plain global reductions."""
import numpy as np
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tex_size,heightmap", [(1, 0), (3, 8), (16, 8), (17, 0), (300, 0)])
@pytest.mark.parametrize("n", [97, (1 << 18) + 5])
def test_copies_agree_with_global_reductions(tex_size, heightmap, n):
    S = lt.Scene(I.box_scene(48, tex_size=tex_size, heightmap=heightmap))
    dI = torch.tensor(I.smooth_adjoint(S.W, S.H, 5), dtype=torch.float32, device="cuda")
    kw = dict(seed=4, n_paths=n, max_depth=8)
    state = S.new_lrb3_state(n)
    grads = {}
    for scatter in (0, 2):
        for accumulate in (False, True):
            S.primal(S.opts(lrb3_state=state, **kw))
            g = S.new_grads()
            g[0].fill_(0.5)
            S.backward_lrb3(S.opts(lrb3_state=state, lrb3_mask_ready=1, scatter=scatter, **kw), dI, grads=g,
                            accumulate=accumulate)
            grads[scatter, accumulate] = g[0].double().cpu().numpy()
    o = S.opts(**kw)
    buf = torch.empty(S.lrb2_buffer_bytes(o), dtype=torch.uint8, device="cuda")
    S.primal(o, estimator=lt.EST_BUFFERED, aux=buf)
    lrb2 = S.backward_lrb2(o, dI, buf)[0].double().cpu().numpy()
    S.sync_status()
    ref = grads[2, False]
    scale = np.linalg.norm(ref)
    # FP32 sums of the same terms in another order (1e-5 as for the scatter modes)
    assert np.linalg.norm(grads[0, False] - ref) < 1e-5 * scale
    assert np.linalg.norm(lrb2 - ref) < 1e-5 * scale
    # added to what the caller's array held (0.5), whose FP32 spacing bounds the difference
    assert np.abs(grads[0, True] - grads[2, True]).max() < 2e-7
