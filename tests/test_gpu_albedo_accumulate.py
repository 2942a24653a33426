"""`accumulate` adds the albedo gradient summed over copies to what the caller's array holds."""
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["lrb3", "lrb2"])
@pytest.mark.parametrize("tex_size", [1, 16])
def test_accumulate_adds_to_the_array(method, tex_size):
    S = lt.Scene(I.box_scene(48, tex_size=tex_size, heightmap=8))
    dI = torch.tensor(I.smooth_adjoint(S.W, S.H, 5), dtype=torch.float32, device="cuda")
    n = 20011
    kw = dict(seed=4, n_paths=n, max_depth=8)
    if method == "lrb3":
        state = S.new_lrb3_state(n)
        S.primal(S.opts(lrb3_state=state, **kw))
        o = S.opts(lrb3_state=state, lrb3_mask_ready=1, **kw)
        run = lambda **a: S.backward_lrb3(o, dI, **a)
    else:
        o = S.opts(**kw)
        buf = torch.empty(S.lrb2_buffer_bytes(o), dtype=torch.uint8, device="cuda")
        S.primal(o, estimator=lt.EST_BUFFERED, aux=buf)
        run = lambda **a: S.backward_lrb2(o, dI, buf, **a)
    once = run()
    scale = once[0].abs().max()
    start = scale * torch.linspace(-1, 1, once[0].numel(), device="cuda")
    g = S.new_grads()
    g[0].copy_(start)
    run(grads=g, accumulate=True)
    S.sync_status()
    # each texel of the copies' sum is added to the array by at most 2^10 / 256 = 4 warps: four
    # roundings at the size of the result (2^-24 of at most 2 scale each), and the sums of the two
    # calls differ by the order of their FP32 adds (1e-5, as in the replays' tests)
    err = (g[0].double() - start.double() - once[0].double()).abs().max()
    assert err <= (8 * 2.0 ** -24 + 1e-5) * float(scale)
    assert float((g[0] - start).abs().max()) > 0.5 * float(scale)
