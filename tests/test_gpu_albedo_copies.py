"""The albedo gradient of LRB-3 pass 3 spread over copies: textures of one texel, of sizes that
are no power of two, and too large for copies to fit, against plain global reductions summed over
parts of the path range in FP64 (one FP32 accumulator per texel over the whole range would itself
be off by more than the tolerance: millions of adds to a one-texel texture)."""
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
    kw = dict(seed=4, max_depth=8, n_norm=n)
    state = S.new_lrb3_state(n)

    def backward(scatter, off, cnt, accumulate=False):
        S.primal(S.opts(lrb3_state=state, path_offset=off, n_paths=cnt, **kw))
        g = S.new_grads()
        if not accumulate:
            g[0].fill_(0.5)  # overwritten
        S.backward_lrb3(S.opts(lrb3_state=state, lrb3_mask_ready=1, scatter=scatter, path_offset=off, n_paths=cnt, **kw),
                        dI, grads=g, accumulate=accumulate)
        return g[0].double().cpu().numpy()

    parts = np.linspace(0, n, 65 if n > 1000 else 2).astype(int)
    ref = sum(backward(2, int(a), int(b - a)) for a, b in zip(parts[:-1], parts[1:]))
    o = S.opts(n_paths=n, **kw)
    buf = torch.empty(S.lrb2_buffer_bytes(o), dtype=torch.uint8, device="cuda")
    S.primal(o, estimator=lt.EST_BUFFERED, aux=buf)
    lrb2 = S.backward_lrb2(o, dI, buf)[0].double().cpu().numpy()
    S.sync_status()
    scale = np.linalg.norm(ref)
    # FP32 sums of the same terms in another order (1e-5 as for the scatter modes)
    assert np.linalg.norm(backward(0, 0, n) - ref) < 1e-5 * scale
    assert np.linalg.norm(backward(0, 0, n, True) - ref) < 1e-5 * scale
    assert np.linalg.norm(lrb2 - ref) < 1e-5 * scale
